"""Kernel edges: sizes at which a kernel changes its layout, word count or path."""
import os

import numpy as np
import pytest

import oracle
from paper_2511_20317_gb300 import tfg
from paper_2511_20317_gb300.tfg import WALKER_INFO_DTYPE
from paper_2511_20317_gb300.workloads import naive_start
from test_gpu_walk import THREADS, assert_parity, gpu  # noqa: F401  (gpu: the module's set-up fixture)

pytestmark = pytest.mark.gpu


def _up(x):
    return (x + 255) // 256 * 256


@pytest.mark.parametrize("fmt", [(4, 5, 5), (5, 6, 9)])
def test_verify_sums_beyond_8_bits(fmt):
    """Eq. (1) on the device when an entry's partial sums leave 8 bits: 130 copies of
    a term followed by 130 of its negative cancel (valid), one more copy does not;
    a checkpoint blob carries the planted best schemes (three 64-bit words per sign)."""
    n, extra = 6, 262
    start = naive_start(*fmt)
    r0 = start.shape[0]
    W = tfg.Walkers([(fmt, 0, start, n)], seed=1, params=tfg.tfg_default_params(r_slack=extra))
    blob = np.frombuffer(W.checkpoint(), dtype=np.uint8).copy()
    info = blob[: n * WALKER_INFO_DTYPE.itemsize].view(WALKER_INFO_DTYPE)
    R = W.pop[0]["r_max"]
    per = R * 2 * 3 * 8
    off = _up(n * WALKER_INFO_DTYPE.itemsize) + _up(n * per)
    best = blob[off: off + n * per].view(np.uint64).reshape(n, R, 2, 3)
    for w, (plus, minus) in enumerate([(130, 130), (131, 130), (130, 131), (0, 0), (127, 127), (1, 0)]):
        t = best[w, 3].copy()                      # one of the naive terms
        neg = t.copy()
        neg[1, 2], neg[0, 2] = t[0, 2], 0          # w negated
        best[w, r0: r0 + plus] = t
        best[w, r0 + plus: r0 + plus + minus] = neg
        info["best_r"][w] = r0 + plus + minus
    W.restore(blob.tobytes())
    assert W.verify_all() == 3                     # the walkers with one copy too many
    W.close()


@pytest.mark.parametrize("mode", [tfg.TFG_MODE_ZT, tfg.TFG_MODE_Z2])
@pytest.mark.parametrize("fmt,slack,nw,policy", [
    ((2, 2, 2), 3, 45, 0), ((2, 3, 4), 8, 60, 0),                         # rows, 32-bit terms, 32 slots
    ((1, 5, 5), 7, 40, 0), ((1, 5, 5), 8, 70, 0),                         # 64-bit terms, 32 and 33 slots
    ((3, 4, 5), 4, 40, 0), ((3, 4, 5), 5, 33, 1), ((3, 3, 4), 28, 40, 1),  # 64 and 65 slots; 64 in use
    ((4, 4, 5), 8, 50, 0), ((4, 4, 5), 8, 33, 2),                         # 88 slots
    ((4, 4, 5), 3, 20001, 0), ((3, 3, 4), 6, 45001, 1),                   # more than reside at once: terms in device memory
])
def test_class_walker_edges(fmt, slack, nw, policy, mode):
    """The thread-per-walker kernel at the edges of its slot words (32 / 33, 64 / 65,
    88 slots), both places of the packed terms, the three walk policies."""
    start = naive_start(*fmt)
    if mode == tfg.TFG_MODE_Z2:
        start = np.abs(start).astype(np.int8)
    steps, L = (700, 120) if nw < 1000 else (400, 120)
    kw = dict(plateau_len=L if policy == 0 else 10**6, walk_policy=policy, r_slack=slack,
              expand_thresh=int(0.03 * 2**32) if policy == 1 else 0)
    W = tfg.Walkers([(fmt, mode, start, nw)], seed=12, params=tfg.tfg_default_params(mapping=1, **kw))
    W.walk(steps // 3).walk(steps - steps // 3).sync()
    take = np.unique(np.linspace(0, nw - 1, 40).astype(int))
    rows = [W.read_walkers(int(w), 1) for w in take]
    info, slots, best = (np.concatenate([x[k] for x in rows]) for k in range(3))
    ref = oracle.Walkers(fmt, start, take, seed=12, mode=mode, plateau_len=kw["plateau_len"], r_slack=slack, policy=policy,
                         expand_thresh=kw["expand_thresh"]).walk(steps, THREADS)
    assert (ref.info["accepted"] > 0).any()
    assert_parity(info, slots, best, ref, range(take.size), f"{fmt} slack {slack} policy {policy} mode {mode}")
    assert W.verify_all() == 0
    W.close()


@pytest.mark.parametrize("nw", [1, 255, 257, 70001])
def test_stats_equal_the_records(nw):
    """Counters, extremes and histogram against the records themselves, below, at and
    above one block of records and beyond the launch's blocks."""
    W = tfg.Walkers([((2, 2, 2), 1, naive_start(2, 2, 2), nw)], seed=4, params=tfg.tfg_default_params(plateau_len=100))
    W.walk(300).sync()
    info, _, _ = W.read_walkers(0, nw, slots=False, best=False)
    st, hist = W.stats(0, hist_len=64)
    assert st["walkers"] == nw and st["steps"] == info["t"].sum()
    for k in ("accepted", "rejected", "nocand", "drops", "merges", "plus", "reductions"):
        assert st[k] == info[k].sum(), k
    assert st["min_best_r"] == info["best_r"].min() and st["max_best_r"] == info["best_r"].max()
    assert np.array_equal(hist, np.bincount(info["best_r"], minlength=64)[:64])
    W.close()


@pytest.mark.parametrize("fmt,slack,nw,horizon", [((2, 2, 2), 3, 33, 1), ((3, 3, 3), 5, 64, 8), ((1, 5, 5), 8, 70, 1),
                                                  ((3, 4, 5), 4, 40, 16), ((3, 4, 5), 5, 65, 1), ((4, 4, 5), 8, 40, 2),
                                                  ((4, 4, 4), 3, 25001, 1)])
def test_uniform_window_steps_in_one_launch(fmt, slack, nw, horizon):
    """Uniform window steps run together equal the same steps called one at a time (a
    window kernel and an apply kernel each): state, choices and the log, at the edges
    of the slot words and with the terms in shared and in device memory."""
    steps = 24 if nw > 1000 else 150
    p = tfg.tfg_default_params(plateau_len=60, r_slack=slack)
    A, B = (tfg.Walkers([(fmt, 0, naive_start(*fmt), nw)], seed=8, params=p) for _ in range(2))
    logs = [tfg.TransitionLog(nw * steps, neg_thresh=int(0.05 * 2**32), horizon=horizon) for _ in range(2)]
    ca = A.walk_window(steps, policy=0, record_choices=True, log=logs[0])
    cb = [B.walk_window(1, policy=0, record_choices=True, log=logs[1]) for _ in range(steps)]
    A.sync()
    assert np.array_equal(ca.cpu().numpy(), np.concatenate([c.cpu().numpy() for c in cb]))
    take = np.unique(np.linspace(0, nw - 1, 64).astype(int))
    ia, ib = (W.read_walkers(0, nw, slots=False, best=False)[0] for W in (A, B))
    assert np.array_equal(ia, ib)
    for w in take:
        for a, b in zip(A.read_walkers(int(w), 1)[1:], B.read_walkers(int(w), 1)[1:]):
            assert np.array_equal(a, b), w
    ea, eb = (np.sort(log.read(), order=["walker_id", "step", "label"]) for log in logs)
    assert len(ea) > 0 and np.array_equal(ea, eb)
    assert np.array_equal(A.window_buffers()[2].cpu().numpy(), B.window_buffers()[2].cpu().numpy())   # last step's sizes
    A.close()
    B.close()


@pytest.mark.parametrize("net", ["random", "zero", "nan"])
@pytest.mark.parametrize("nw", [1, 33, 200])
def test_greedy_choice_is_the_first_best_row(nw, net):
    """The learned policy's choice: the first row of highest score among the window's K,
    in full and partial warps; with a network of zeros every score ties; NaN scores
    compare false, so row 0 stays chosen when every score is one."""
    import torch
    from paper_2511_20317_gb300 import learned
    fmt = (3, 4, 5)
    W = tfg.Walkers([(fmt, 0, naive_start(*fmt), nw)], seed=6, params=tfg.tfg_default_params(plateau_len=500))
    W.walk(150)
    params = learned.init_params(3)
    if net != "random":
        params.zero_()
    if net == "nan":
        params[-16:-12].view(torch.float32).fill_(float("nan"))   # b3
    ch = W.walk_window(1, policy=1, mlp_params=params, record_choices=True).cpu().numpy()[0]
    W.sync()
    _, score, K = (b.cpu().numpy() for b in W.window_buffers())
    for w in range(nw):
        s = score[w, : K[w]]
        want = 0 if np.isnan(s[0]) else int(np.nanargmax(s))
        assert ch[w] == want, w
    W.close()


@pytest.mark.parametrize("fmt,slack,steps", [((2, 2, 2), 3, 50), ((3, 3, 3), 5, 0), ((1, 5, 5), 8, 60), ((3, 4, 5), 6, 400),
                                             ((4, 4, 4), 3, 300), ((4, 4, 5), 8, 500)])
def test_window_rows_equal_the_oracle(fmt, slack, steps):
    """Window rows and sizes at 1, 2 and 3 chunks of slots, full and sparse windows, on
    walked states, against the oracle's window."""
    nw = 40
    W = tfg.Walkers([(fmt, 0, naive_start(*fmt), nw)], seed=2, params=tfg.tfg_default_params(plateau_len=40, r_slack=slack))
    W.walk(steps).sync()
    info, slots, _ = W.read_walkers(0, nw)
    _, rows, sizes = W.window_dump(features=False)
    rows, sizes = rows.cpu().numpy(), sizes.cpu().numpy()
    for w in range(nw):
        r, t = int(info["r"][w]), int(info["t"][w])
        i0 = (int(oracle.philox4x32_10([t, 0, w, 0], [2, 0])[0]) * r) >> 32
        feat, cand = oracle.window_features(fmt, slots[w, :r], int(info["best_r"][w]), i0)
        assert sizes[w] == len(cand), w
        d, i = rows[w, : sizes[w], 0].view(np.uint32), rows[w, : sizes[w], 1]
        got = np.stack([d & 1023, (d >> 10) & 3, (d >> 12) & 1023, np.where((d >> 22) & 1, -1, 1), (d >> 23) & 1], 1)
        assert np.array_equal(got, cand), w
        assert np.array_equal(i & 255, feat[:, 18]) and np.array_equal(i >> 8, feat[:, 24]), w
    W.close()


@pytest.mark.parametrize("mode", [tfg.TFG_MODE_ZT, tfg.TFG_MODE_Z2])
@pytest.mark.parametrize("fmt,slack,nw,policy", [
    ((4, 5, 5), 3, 300, 0), ((4, 5, 5), 6, 301, 1),                            # every step searching
    ((4, 5, 5), 28, 4003, 0), ((4, 5, 5), 29, 5001, 0),                        # kept classes: 128 / 129 slots
    ((4, 5, 5), 3, 20003, 0), ((4, 5, 5), 6, 8003, 1), ((4, 5, 5), 28, 8001, 1), ((4, 5, 5), 2, 9001, 2),
    ((9, 8, 2), 3, 4801, 0), ((9, 1, 8), 3, 8001, 2), ((9, 8, 2), 5, 8003, 1),  # two words per factor
])
def test_wide_walker_edges(fmt, slack, nw, policy, mode):
    """The wide-term kernels on both sides of the choice between them, at the edges of the
    hash words, with the last warp partly filled, the terms in shared and in device memory,
    the walk policies."""
    start = naive_start(*fmt)
    if mode == tfg.TFG_MODE_Z2:
        start = np.abs(start).astype(np.int8)
    steps = 320
    kw = dict(plateau_len=60 if policy == 0 else 10**6, walk_policy=policy, r_slack=slack,
              expand_thresh=int(0.03 * 2**32) if policy == 1 else 0)
    W = tfg.Walkers([(fmt, mode, start, nw)], seed=13, params=tfg.tfg_default_params(**kw))
    if policy:
        W.walk(steps).sync()
    else:
        W.walk(steps // 3).walk(steps - steps // 3).sync()
    take = np.unique(np.concatenate([np.linspace(0, nw - 1, 16).astype(int), np.arange(max(0, nw - 5), nw)]))
    rows = [W.read_walkers(int(w), 1) for w in take]
    info, slots, best = (np.concatenate([x[k] for x in rows]) for k in range(3))
    ref = oracle.Walkers(fmt, start, take, seed=13, mode=mode, plateau_len=kw["plateau_len"], r_slack=slack, policy=policy,
                         expand_thresh=kw["expand_thresh"]).walk(steps, THREADS)
    assert (ref.info["accepted"] > 0).any()
    assert_parity(info, slots, best, ref, range(take.size), f"{fmt} slack {slack} policy {policy} mode {mode}")
    assert W.verify_all() == 0
    W.close()


@pytest.mark.parametrize("n,shift", [(1, 0), (127, 1), (129, 0), (128 * 152 + 1, 0), (128 * 152 * 2 + 77, 1),
                                     (128 * 152 * 3 + 5, 0)])
def test_gradient_tiles_and_warpgroups(n, shift):
    """Gradient sums at the edges of the tiles and of the two warpgroups' shares, the
    parameters at a 16-byte or (shift) only 4-byte boundary, single launch and training
    step, against the float64 reference.  Bound per entry: one bf16 ulp (2^-8) on each
    operand of every product term, plus FP32 sum error."""
    import torch
    from oracle import mlp
    rng = np.random.default_rng(n)
    p = mlp.Params.random(rng)
    x = rng.integers(0, 9, size=(n, mlp.IN)).astype(np.float32)
    x[:, 24:] = mlp.bf16_round(rng.normal(0, 1, size=(n, mlp.IN - 24)))
    label = (rng.random(n) < 0.3).astype(np.float32)
    weight = (rng.random(n) / n).astype(np.float32)
    y, cache = mlp.forward(p, x)
    loss, dy = mlp.logistic_loss(y, label, weight)
    ref = mlp.backward(p, cache, dy, bf16_operands=True)
    blob = np.frombuffer(p.blob(), dtype=np.uint8)
    room = torch.zeros(blob.size + 16, dtype=torch.uint8, device="cuda")
    params = room[4 * shift:4 * shift + blob.size]
    params.copy_(torch.from_numpy(blob.copy()))
    xs = torch.from_numpy(mlp.bf16_bits(mlp.bf16_round(x)).view(np.int16).copy()).cuda().view(torch.bfloat16)
    ls, ws = torch.from_numpy(label).cuda(), torch.from_numpy(weight).cuda()
    P = tfg.MLP_NUM_PARAMS
    g, gloss = tfg.tfg_mlp_grad(params, xs, ls, ws)
    tr = tfg.MlpTrainer(params)
    tr.step(xs, ls, ws, 0.0)
    state = tr.state[3 * P:4 * P + 1].cpu().numpy()
    for vec, total in ((g.cpu().numpy(), gloss), (state[:P], state[P])):
        assert abs(total - loss) <= 1e-4 * (1 + abs(loss))
        got = mlp.split_vector(vec.astype(np.float64))
        for name in ["W1", "W2", "b1", "b2", "w3", "b3"]:
            bound = 2.0 ** -7 * np.asarray(ref["_abs"][name]) + 1e-6 * (1 + np.abs(ref[name]))
            diff = np.abs(np.asarray(got[name]) - np.asarray(ref[name]))
            assert (diff <= bound).all(), (name, float(np.max(diff - bound)))


@pytest.mark.parametrize("fmt,nw", [((2, 2, 2), 5), ((2, 2, 3), 40009), ((3, 3, 3), 20011)])
def test_window_scores_of_ragged_windows(fmt, nw):
    """Scores of every window row, windows of all sizes laid end to end in groups of 32 rows and
    many windows to a warpgroup, against the network on the dumped features (float32
    products of the same bf16 operands).  Bound as for row scoring: two bf16 flips of a
    hidden unit a row, 2 * 2^-8 * max_h |h1_h| sum_o |W2[h,o] w3[o]|, plus FP32 sums."""
    import torch
    from oracle import mlp
    W = tfg.Walkers([(fmt, 0, naive_start(*fmt), nw)], seed=3, params=tfg.tfg_default_params(plateau_len=100))
    W.walk_window(200, policy=0)
    feat, _, kwin = W.window_dump()
    feat, kwin = feat.clone(), kwin.clone()
    p = mlp.Params.random(np.random.default_rng(6))
    blob = torch.from_numpy(np.frombuffer(p.blob(), dtype=np.uint8).copy()).cuda()
    W.walk_window(1, policy=1, mlp_params=blob)
    W.sync()
    _, score, kwin2 = W.window_buffers()
    assert torch.equal(kwin, kwin2) and (nw < 100 or kwin.unique().numel() > 1)
    W1, W2, b1, b2, w3 = (torch.from_numpy(np.asarray(a, np.float32)).cuda() for a in (p.W1, p.W2, p.b1, p.b2, p.w3))
    path = W2.abs() @ w3.abs()
    for lo in range(0, nw, 4096):
        rows = torch.arange(256, device="cuda")[None] < kwin[lo:lo + 4096, None]
        x = feat[lo:lo + 4096][rows].float()
        h1 = torch.relu(x.double() @ W1.double() + b1.double()).float().bfloat16().float()
        y = torch.relu(h1.double() @ W2.double() + b2.double()) @ w3.double() + float(p.b3)
        bound = 2 * ((h1.abs() * 2.0 ** -8) * path).amax(1) + 1e-5 * (1 + y.abs())
        assert ((score[lo:lo + 4096][rows].double() - y).abs() <= bound).all()
    W.close()


@pytest.mark.parametrize("fmt,nw,policy", [((2, 3, 4), 60001, 0), ((2, 3, 4), 60001, 1), ((2, 3, 4), 60001, 2),
                                           ((2, 3, 3), 70001, 0), ((3, 3, 3), 70001, 0), ((3, 3, 3), 19456, 0),
                                           ((3, 3, 3), 19457, 0), ((3, 3, 3), 20033, 2), ((2, 2, 6), 60001, 0)])
@pytest.mark.parametrize("mode", [0, 1])
def test_populations_at_which_the_class_walker_changes(fmt, nw, policy, mode):
    """Populations on either side of the choice between factor classes as rows and as lists (two
    waves of rows against one of lists; short factors keep rows) and between bit
    slices and classes, walkers spread over the population against the oracle."""
    L, steps = 40, 400
    start = naive_start(*fmt)
    kw = dict(plateau_len=L if policy == 0 else 10**6, walk_policy=policy,
              expand_thresh=int(0.03 * 2**32) if policy == 1 else 0)
    W = tfg.Walkers([(fmt, mode, start, nw)], seed=14, params=tfg.tfg_default_params(**kw))
    W.walk(steps).sync()
    take = np.linspace(0, nw - 1, 48).astype(int)
    rows = [W.read_walkers(int(w), 1) for w in take]
    info, slots, best = (np.concatenate([x[k] for x in rows]) for k in range(3))
    ref = oracle.Walkers(fmt, start, take, seed=14, mode=mode, plateau_len=kw["plateau_len"], policy=policy,
                         expand_thresh=kw["expand_thresh"])
    ref.walk(steps, threads=THREADS)
    assert_parity(info, slots, best, ref, range(take.size), f"{fmt} {nw} policy {policy} mode {mode}")
    W.close()


@pytest.mark.parametrize("nw", [1, 1217, 2433, 4865, 9729])
@pytest.mark.parametrize("fmt,mode,policy", [((2, 2, 2), 0, 0), ((2, 3, 4), 1, 1), ((3, 3, 3), 0, 0), ((3, 3, 3), 1, 0),
                                             ((2, 3, 3), 0, 2), ((4, 4, 5), 0, 0), ((4, 4, 5), 1, 2)])
def test_small_populations_in_few_lanes(fmt, mode, policy, nw):
    """Populations of which a warp takes 1, 2, 4, 8 or 16 walkers (a block's last lanes empty),
    alone and beside another population, against the oracle: the walkers at both ends and spread between."""
    L, steps = 60, 300
    start = naive_start(*fmt)
    kw = dict(plateau_len=L if policy == 0 else 10**6, walk_policy=policy,
              expand_thresh=int(0.03 * 2**32) if policy == 1 else 0)
    other = [((2, 2, 3), 0, naive_start(2, 2, 3), 77)] if nw < 5000 else []
    W = tfg.Walkers([(fmt, mode, start, nw)] + other, seed=15, params=tfg.tfg_default_params(**kw))
    W.walk(steps // 2).walk(steps - steps // 2).sync()
    take = np.unique(np.concatenate([np.arange(min(nw, 8)), np.linspace(0, nw - 1, 24).astype(int),
                                     np.arange(max(0, nw - 8), nw)]))
    rows = [W.read_walkers(int(w), 1) for w in take]
    info, slots, best = (np.concatenate([x[k] for x in rows]) for k in range(3))
    ref = oracle.Walkers(fmt, start, take, seed=15, mode=mode, plateau_len=kw["plateau_len"], policy=policy,
                         expand_thresh=kw["expand_thresh"])
    ref.walk(steps, threads=THREADS)
    assert_parity(info, slots, best, ref, range(take.size), f"{fmt} {nw} policy {policy} mode {mode}")
    assert W.verify_all() == 0
    W.close()


@pytest.mark.parametrize("fmt,nw", [((2, 2, 2), 301), ((3, 4, 5), 1217), ((4, 4, 4), 2433), ((2, 3, 3), 4865)])
def test_uniform_window_walk_in_few_lanes(fmt, nw):
    """The joint launch of uniform window steps on small populations equals the same steps
    one by one, walker records and choices."""
    steps = 12
    mk = lambda: tfg.Walkers([(fmt, 0, naive_start(*fmt), nw)], seed=16, params=tfg.tfg_default_params(plateau_len=50))
    A, B = mk(), mk()
    ca = A.walk_window(steps, policy=0, record_choices=True)
    cb = [B.walk_window(1, policy=0, record_choices=True) for _ in range(steps)]
    A.sync(), B.sync()
    assert np.array_equal(ca.cpu().numpy(), np.concatenate([c.cpu().numpy() for c in cb]))
    for x, y in zip(A.read_walkers(0, nw), B.read_walkers(0, nw)):
        assert np.array_equal(x, y)
    A.close(), B.close()


def test_timeout_reaches_the_host_error_word():
    """A completion wait that gives up raises from the call that made its own error word (in
    host memory), and the next call is clean."""
    import torch
    from oracle import mlp
    p = mlp.Params.random(np.random.default_rng(2))
    blob = torch.from_numpy(np.frombuffer(p.blob(), dtype=np.uint8).copy()).cuda()
    x = torch.zeros((1000, 32), dtype=torch.bfloat16, device="cuda")
    want = tfg.tfg_mlp_score(blob, x)
    tfg.tfg_test_set_wait_limit(0)
    try:
        with pytest.raises(tfg.TfgError):
            tfg.tfg_mlp_score(blob, x)
    finally:
        tfg.tfg_test_set_wait_limit(-1)
    assert torch.equal(tfg.tfg_mlp_score(blob, x), want)


@pytest.mark.parametrize("fmt,nw", [((2, 2, 2), 5), ((4, 4, 5), 33)])
def test_window_dump_rows_at_an_8_byte_boundary(fmt, nw):
    """The dump takes descriptors at any 8-byte boundary: the same rows and sizes as at a
    16-byte one, nothing written before, after or past a window."""
    import ctypes
    import torch
    W = tfg.Walkers([(fmt, 0, naive_start(*fmt), nw)], seed=5, params=tfg.tfg_default_params(plateau_len=100))
    W.walk(200)
    _, want, sizes = W.window_dump(features=False)
    words = nw * tfg.WINDOW * 2
    room = torch.full((words + 8,), -7, dtype=torch.int32, device="cuda")
    kwin = torch.zeros(nw, dtype=torch.int32, device="cuda")
    assert room.data_ptr() % 16 == 0
    rc = tfg.lib().tfg_window_dump(W.ctx, None, ctypes.c_void_p(room.data_ptr() + 8), ctypes.c_void_p(kwin.data_ptr()))
    assert rc == tfg.TFG_OK
    W.sync()
    got = room[2:2 + words].view(nw, tfg.WINDOW, 2)
    inside = (torch.arange(tfg.WINDOW, device="cuda")[None, :, None] < sizes[:, None, None]).expand(-1, -1, 2)
    assert torch.equal(kwin, sizes) and torch.equal(got[inside], want[inside]) and (got[~inside] == -7).all()
    assert (room[:2] == -7).all() and (room[2 + words:] == -7).all()
    W.close()


def _raised_start(fmt, seed=3):
    """A scheme two expansions above the naive one, which walks without expansions come down from."""
    W = tfg.Walkers([(fmt, 0, naive_start(*fmt), 64)], seed=seed, params=tfg.tfg_default_params(plateau_len=2))
    W.walk(8).sync()
    info, slots, _ = W.read_walkers(0, 64)
    W.close()
    w = int(np.argmax(info["r"]))
    assert info["r"][w] > naive_start(*fmt).shape[0]
    return slots[w, : info["r"][w]]


@pytest.mark.parametrize("mapping", [1, 32])
@pytest.mark.parametrize("fmt,mode", [((2, 2, 3), 0), ((2, 3, 4), 1), ((3, 3, 4), 0), ((3, 3, 4), 1)])
@pytest.mark.parametrize("L", [2**63 - 1, 2**63 - 700])
def test_plateaus_beyond_the_step_counter(fmt, mode, L, mapping):
    """A plateau length of 2^63 - 1 (never) and one just below: no expansion, over launches that
    start before and after the first better scheme, with every kind of mapping."""
    start, nw, steps = _raised_start(fmt), 70, 1800
    if mode:
        start = np.abs(start).astype(np.int8)
    W = tfg.Walkers([(fmt, mode, start, nw)], seed=18, params=tfg.tfg_default_params(plateau_len=L, mapping=mapping))
    for part in (40, 760, 1000):
        W.walk(part)
    W.sync()
    info, slots, best = W.read_walkers(0, nw)
    ref = oracle.Walkers(fmt, start, np.arange(nw), seed=18, mode=mode, plateau_len=L).walk(steps, THREADS)
    assert (ref.info["plus"] == 0).all() and (ref.info["best_t"] > 0).any()
    assert_parity(info, slots, best, ref, range(nw), f"{fmt} mode {mode} plateau {L}")
    W.close()


def test_uniform_window_walk_without_plateaus():
    """The joint launch of uniform window steps with a plateau length of 2^63 - 1."""
    fmt, nw, steps, L = (3, 3, 4), 70, 900, 2**63 - 1
    start = _raised_start(fmt)
    W = tfg.Walkers([(fmt, 0, start, nw)], seed=19, params=tfg.tfg_default_params(plateau_len=L))
    for part in (400, 500):
        W.walk_window(part, policy=0)
    W.sync()
    info, slots, best = W.read_walkers(0, nw)
    ref = oracle.Walkers(fmt, start, np.arange(nw), seed=19, plateau_len=L).walk_window(steps)
    assert (ref.info["plus"] == 0).all() and (ref.info["best_t"] > 0).any()
    assert_parity(info, slots, best, ref, range(nw), "window")
    W.close()


@pytest.mark.parametrize("b2", [np.inf, -np.inf, 3.4e38, -3.4e38, 1e-3])
def test_scores_with_an_extreme_bias(b2):
    """An output bias of the second layer that is infinite, or finite beyond the largest BF16 value:
    the score is the FP32 sum's.  Bound: the FP32 sum of 128 products and the bf16 flip of
    a hidden unit, as for row scoring."""
    import torch
    from oracle import mlp
    rng = np.random.default_rng(4)
    p = mlp.Params.random(rng)
    unit = 5
    p.w3[unit] = np.float32(1e-32 if np.isfinite(b2) and abs(b2) > 1 else 0.5)
    p.b2[unit] = np.float32(b2)
    x = mlp.bf16_round(rng.integers(0, 9, size=(300, mlp.IN)).astype(np.float32))
    y, _ = mlp.forward(p, x)
    blob = torch.from_numpy(np.frombuffer(p.blob(), dtype=np.uint8).copy()).cuda()
    xs = torch.from_numpy(mlp.bf16_bits(x).view(np.int16).copy()).cuda().view(torch.bfloat16)
    got = tfg.tfg_mlp_score(blob, xs).cpu().numpy().astype(np.float64)
    if np.isinf(y).any():
        assert np.isinf(y).all() and np.array_equal(got, y)
        return
    z1 = mlp.bf16_round(x).astype(np.float64) @ p.W1 + p.b1
    h1 = np.maximum(mlp.bf16_round(np.maximum(z1, 0)), 0).astype(np.float64)
    path = np.abs(p.W2) @ np.abs(p.w3)
    bound = 2 * ((h1 * 2.0 ** -8) * path).max(1) + 1e-5 * (1 + np.abs(y))
    assert (np.abs(got - y) <= bound).all()


def test_verification_from_two_threads():
    """Two threads verify populations whose accumulators need different shared memory by the same
    kernel: no call fails."""
    import threading
    import torch
    from paper_2511_20317_gb300 import starts
    errors = []
    walkers = []
    for fmt, start in (((6, 7, 9), starts.start_6_7_9()[1]), ((5, 5, 5), naive_start(5, 5, 5))):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            walkers.append((tfg.Walkers([(fmt, 0, start, 2)], seed=1, stream=st), torch.zeros(1, dtype=torch.int64, device="cuda")))
    torch.cuda.synchronize()

    def verify(W, fails):
        import ctypes
        torch.cuda.set_device(0)
        for _ in range(2000):
            if tfg.lib().tfg_verify_all_async(W.ctx, ctypes.c_void_p(fails.data_ptr())) != tfg.TFG_OK:
                errors.append(tfg.lib().tfg_last_error())
                return

    threads = [threading.Thread(target=verify, args=a) for a in walkers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    assert all(int(f.item()) == 0 for _, f in walkers)
    for W, _ in walkers:
        W.close()


def test_resizes_from_two_threads():
    """Two threads resize into populations whose terms need different shared memory: no call fails."""
    import threading
    import torch
    errors, jobs = [], []
    for src, dst, aux in (((2, 2, 2), (2, 2, 3), None), ((1, 1, 1), (8, 9, 9), (8, 9, 9))):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            W = tfg.Walkers([(src, 0, naive_start(*src), 4), (dst, 0, naive_start(*dst), 4)], seed=1, stream=st)
        jobs.append((W, aux))
    torch.cuda.synchronize()

    def resize(W, aux):
        torch.cuda.set_device(0)
        try:
            for _ in range(1000):
                if aux:
                    skipped = W.resize(tfg.TFG_RESIZE_PRODUCT, 0, 4, 4, aux=(aux, naive_start(*aux)))
                else:
                    skipped = W.resize(tfg.TFG_RESIZE_EXTEND, 0, 4, 4, axis=2)
                assert skipped == 0
        except Exception as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=resize, args=a) for a in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for W, _ in jobs:
        assert W.verify_all() == 0
        W.close()


def test_a_full_log_keeps_the_earliest_steps():
    """A log that fills up during uniform window steps of more walkers than reside at once: no entry
    is of a step 256 or more after one that is lost.  A sixteenth of the steps is kept
    (3750 a step, standard deviation 59; a step of which a tenth is missing counts as lost)."""
    fmt, nw, steps = (4, 4, 4), 60001, 640
    W = tfg.Walkers([(fmt, 0, naive_start(*fmt), nw)], seed=20, params=tfg.tfg_default_params(plateau_len=10**6))
    W.walk(100)
    log = tfg.TransitionLog(nw * 240 // 16, neg_thresh=2**28)
    W.walk_window(steps, policy=0, log=log)
    W.sync()
    e = log.read()
    assert len(e) == log.capacity < int(log.count.item())
    kept = np.bincount(e["step"] - 100, minlength=steps)
    lost = int(np.argmax(kept < 0.9 * nw / 16))
    assert lost >= 128 and (kept[lost + 256:] == 0).all()
    W.close()


def _launches(call):
    """(name, threads per block, blocks) of the walk kernels that call() launches."""
    import json
    import tempfile
    import torch
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]):   # a process's first session may miss launches
        torch.zeros(1, device="cuda").add_(1)
        torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    with tempfile.TemporaryDirectory() as d:
        prof.export_chrome_trace(os.path.join(d, "trace.json"))
        with open(os.path.join(d, "trace.json")) as f:
            events = json.load(f)["traceEvents"]
    out = [(e["name"], int(np.prod(e["args"]["block"])), int(np.prod(e["args"]["grid"])))
           for e in events if e.get("cat") == "kernel" and "walk_" in e["name"]]
    if not out:
        pytest.skip("no kernel records from the profiler here")
    return out


@pytest.mark.parametrize("fmt,block,mode", [((3, 3, 4), 96, 0), ((3, 4, 5), 128, 0), ((4, 4, 4), 128, 0), ((4, 4, 5), 160, 0),
                                            ((4, 4, 5), 64, 0), ((4, 4, 5), 128, 1), ((3, 3, 3), 64, 0)])
@pytest.mark.parametrize("nw", [700, 20001])
def test_walkers_per_block_that_were_asked_for(fmt, block, mode, nw):
    """block_threads that name a compiled choice are the walkers per block of the launch itself,
    also of a population that would otherwise spread over more warps, and change no walk."""
    start, steps, L = naive_start(*fmt), 400, 60
    if mode:
        start = np.abs(start).astype(np.int8)
    W = tfg.Walkers([(fmt, mode, start, nw)], seed=21,
                    params=tfg.tfg_default_params(plateau_len=L, mapping=1, block_threads=block, use_graph=0))
    launched = _launches(lambda: W.walk(steps // 4).walk(steps - steps // 4).sync())
    assert {x[1:] for x in launched} == {(block, (nw + block - 1) // block)}
    take = np.unique(np.linspace(0, nw - 1, 40).astype(int))
    rows = [W.read_walkers(int(w), 1) for w in take]
    info, slots, best = (np.concatenate([x[k] for x in rows]) for k in range(3))
    ref = oracle.Walkers(fmt, start, take, seed=21, mode=mode, plateau_len=L).walk(steps, THREADS)
    assert (ref.info["plus"] > 0).any()
    assert_parity(info, slots, best, ref, range(take.size), f"{fmt} block {block}")
    W.close()


@pytest.mark.parametrize("fmt,mode,nw,policy", [
    ((2, 2, 2), 0, 300, 0), ((2, 3, 4), 0, 5001, 0), ((2, 3, 4), 1, 5001, 2), ((2, 3, 4), 0, 70001, 0), ((3, 3, 3), 0, 1001, 0),
    ((3, 3, 3), 0, 10001, 0), ((3, 3, 3), 0, 70001, 0), ((3, 3, 3), 1, 10001, 0), ((2, 4, 4), 0, 1001, 0), ((2, 4, 4), 1, 20001, 0),
    ((4, 4, 5), 0, 1001, 0), ((4, 4, 5), 0, 30001, 0), ((4, 4, 5), 1, 3001, 2), ((4, 5, 5), 0, 301, 0), ((4, 5, 5), 0, 5001, 0),
])
def test_the_launch_shape_is_the_launch(fmt, mode, nw, policy):
    """Threads per block and blocks that population() reports (tfg_launch_shape) are those of the
    walk's launch: small populations, every-slot, bit-sliced, class, lane-group and wide kernels."""
    start = naive_start(*fmt)
    if mode:
        start = np.abs(start).astype(np.int8)
    W = tfg.Walkers([(fmt, mode, start, nw)], seed=22, params=tfg.tfg_default_params(walk_policy=policy, use_graph=0))
    launched = _launches(lambda: W.walk(200).sync())
    assert [x[1:] for x in launched] == [(W.pop[0]["block_threads"], W.pop[0]["grid"])]
    W.close()


@pytest.mark.parametrize("fmt,mode,nw,policy", [((2, 2, 2), 0, 20001, 0), ((2, 3, 4), 0, 70001, 0), ((3, 3, 3), 0, 70001, 0),
                                                ((3, 3, 3), 0, 10001, 1), ((2, 3, 4), 0, 20001, 2), ((4, 4, 5), 0, 30001, 0)])
@pytest.mark.parametrize("graph", [0, 1])
def test_the_autotuner_times_the_kernel_of_the_walk(fmt, mode, nw, policy, graph):
    """A trial on a few of a population's walkers runs the kernel, at the threads per block, that
    the whole population's walk runs before it, and the choice's walk runs one that a trial ran."""
    start = naive_start(*fmt)
    W = tfg.Walkers([(fmt, mode, start, nw)], seed=23, params=tfg.tfg_default_params(walk_policy=policy, use_graph=graph))
    before = _launches(lambda: W.walk(100).sync())
    trials = _launches(lambda: W.autotune(trial_steps=100, trial_walkers=1024))
    after = _launches(lambda: W.walk(100).sync())
    assert trials[0][:2] == before[0][:2] and trials[0][2] == -(-1024 // before[0][1])
    assert after[0][:2] in [x[:2] for x in trials]
    W.close()


def test_the_autotuner_judges_the_whole_population():
    """Sixteen lanes a walker are the fastest on a trial that leaves most of the GPU idle and take 1.4
    times as long as one on the whole population: the choice is one."""
    fmt, nw = (3, 3, 3), 131072
    W = tfg.Walkers([(fmt, 1, np.abs(naive_start(*fmt)).astype(np.int8), nw)], seed=24,
                    params=tfg.tfg_default_params(walk_policy=1, r_slack=6, expand_thresh=int(0.01 * 2**32)))
    W.walk(500).sync()
    assert W.autotune(trial_steps=300, trial_walkers=16384) == [1]
    W.close()


@pytest.mark.parametrize("fmt,mode,nw,policy,slack,kernel", [
    *[((2, 4, 4), mode, nw, policy, 3, kernel) for mode in (0, 1) for nw, policy, kernel in
      ((8193, 0, "walk_link"), (8191, 0, "walk_group"), (8193, 2, "walk_link"), (16385, 1, "walk_link"), (16383, 1, "walk_group"))],
    ((2, 3, 5), 0, 8193, 0, 3, "walk_link"), ((2, 3, 5), 1, 8193, 2, 34, "walk_link"), ((2, 3, 5), 0, 16385, 1, 6, "walk_link"),
    ((3, 3, 4), 1, 60001, 1, 6, "walk_link"), ((4, 4, 5), 1, 45001, 0, 3, "walk_link"),   # terms in device memory
])
def test_default_mapping_of_many_walkers(fmt, mode, nw, policy, slack, kernel):
    """32-bit terms of more than 32 slots on either side of the population from which a thread takes
    a walker by default, and Z_2 populations of more than reside at once, against the oracle."""
    start, steps, L = naive_start(*fmt), 300, 60
    if mode:
        start = np.abs(start).astype(np.int8)
    kw = dict(plateau_len=L if policy == 0 else 10**6, walk_policy=policy, r_slack=slack,
              expand_thresh=int(0.03 * 2**32) if policy == 1 else 0)
    W = tfg.Walkers([(fmt, mode, start, nw)], seed=25, params=tfg.tfg_default_params(use_graph=0, **kw))
    launched = _launches(lambda: W.walk(steps // 2).walk(steps - steps // 2).sync())
    assert all(kernel in x[0] for x in launched) and launched[0][1] == W.pop[0]["block_threads"]
    if nw > 20000:   # the fourth template argument of the kernel: terms in the walker's device-memory slots
        args = launched[0][0].split("<", 1)[1].split(",")
        assert args[3].strip().replace("(bool)", "") in ("1", "true"), launched[0][0]
    take = np.unique(np.concatenate([np.linspace(0, nw - 1, 40).astype(int), np.arange(nw - 4, nw)]))
    rows = [W.read_walkers(int(w), 1) for w in take]
    info, slots, best = (np.concatenate([x[k] for x in rows]) for k in range(3))
    ref = oracle.Walkers(fmt, start, take, seed=25, mode=mode, plateau_len=kw["plateau_len"], r_slack=slack, policy=policy,
                         expand_thresh=kw["expand_thresh"]).walk(steps, THREADS)
    assert (ref.info["accepted"] > 0).any()
    assert_parity(info, slots, best, ref, range(take.size), f"{fmt} {nw} policy {policy} mode {mode}")
    assert W.verify_all() == 0
    W.close()


@pytest.mark.parametrize("fmt,mode,nw,kernel", [((2, 2, 2), 0, 12001, "walk_link"), ((2, 2, 2), 0, 12301, "walk_solo"),
                                                ((2, 2, 3), 1, 2500, "walk_link"), ((2, 2, 3), 1, 6201, "walk_solo"),
                                                ((2, 3, 3), 1, 10001, "walk_link"), ((2, 3, 3), 1, 12301, "walk_solo")])
def test_expansion_policy_on_few_slots(fmt, mode, nw, kernel):
    """Walk policy 1 on the smallest ranks, on either side of the population (walkers an SM) from
    which testing every slot is the faster, against the oracle."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("sizes of a GPU of 152 SMs")
    start, steps = naive_start(*fmt), 300
    if mode:
        start = np.abs(start).astype(np.int8)
    kw = dict(plateau_len=10**6, walk_policy=1, expand_thresh=int(0.03 * 2**32))
    W = tfg.Walkers([(fmt, mode, start, nw)], seed=26, params=tfg.tfg_default_params(use_graph=0, **kw))
    launched = _launches(lambda: W.walk(steps).sync())
    assert kernel in launched[0][0]
    take = np.unique(np.concatenate([np.linspace(0, nw - 1, 40).astype(int), np.arange(nw - 4, nw)]))
    rows = [W.read_walkers(int(w), 1) for w in take]
    info, slots, best = (np.concatenate([x[k] for x in rows]) for k in range(3))
    ref = oracle.Walkers(fmt, start, take, seed=26, mode=mode, plateau_len=10**6, policy=1,
                         expand_thresh=kw["expand_thresh"]).walk(steps, THREADS)
    assert_parity(info, slots, best, ref, range(take.size), f"{fmt} {nw} mode {mode}")
    W.close()


def test_network_calls_take_any_stream_handle():
    """Scores and gradients on a stream given as an object that has only its handle."""
    import types
    import torch
    from oracle import mlp
    p = mlp.Params.random(np.random.default_rng(3))
    blob = torch.from_numpy(np.frombuffer(p.blob(), dtype=np.uint8).copy()).cuda()
    x = torch.ones((300, 32), dtype=torch.bfloat16, device="cuda")
    label = torch.ones(300, device="cuda")
    stream = types.SimpleNamespace(cuda_stream=torch.cuda.current_stream().cuda_stream)
    assert torch.equal(tfg.tfg_mlp_score(blob, x, stream=stream), tfg.tfg_mlp_score(blob, x))
    assert abs(tfg.tfg_mlp_grad(blob, x, label, label, stream=stream)[1] - tfg.tfg_mlp_grad(blob, x, label, label)[1]) < 1e-2
