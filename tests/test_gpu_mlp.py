"""Parity of the duration surrogate's CUDA path (fn_mlp_*) with its FP64
reference (oracle/mlp.py), and of the windowed scan with the full scan."""
import numpy as np
import pytest
import torch

import oracle.mlp as M
from paper_2609_22608_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_2609_22608_gb300 import surrogate
    return surrogate


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def seeded_params(seed):
    rng = np.random.default_rng(seed)
    ps = []
    for l in range(4):
        fi, fo = M.DIMS[l], M.DIMS[l + 1]
        W = rng.normal(0, np.sqrt(2.0 / fi), (fi, fo)).astype(np.float32)
        if l == 0:
            W[28:] = 0
        b = rng.normal(0, 0.05, fo).astype(np.float32)
        ps.append((W, b))
    return ps


def relerr(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-30))


def elementwise_ok(Y, ref):
    """Per output element against the FP64 reference with the same bf16
    rounding points.  The GPU accumulates in FP32 in another order, so a
    hidden activation that sits at a bf16 rounding boundary can round to the
    neighbouring value (one bf16 ulp, 2^-8 relative), which moves an output
    by at most ~1e-2 of the output scale; every element must be within that,
    and 99 % of them within 2e-3 of the scale (no such flip upstream)."""
    Y = np.asarray(Y, np.float64)
    scale = max(1.0, float(np.abs(ref).max()))
    err = np.abs(Y - ref)
    return bool(err.max() <= 1e-2 * scale and np.quantile(err, 0.99) <= 2e-3 * scale), \
        float(err.max() / scale)


def load(mlp, ps):
    for l, (W, b) in enumerate(ps):
        mlp.set_params(l, W, b)


def test_forward_parity(S, arm):
    mlp = S.MLP(max_batch=1024)
    ps = seeded_params(0)
    load(mlp, ps)
    s0, s1 = synth.random_edges(arm, 700, 3)
    Y = mlp.predict(arm, dev(s0), dev(s1)).cpu().numpy()
    ref, _ = M.forward([(W.astype(np.float64), b.astype(np.float64)) for W, b in ps],
                       M.features(arm, s0, s1))
    assert relerr(Y, ref) < 1e-3
    ok, worst = elementwise_ok(Y, ref)
    assert ok, worst
    mlp.close()


@pytest.mark.parametrize("E", [1, 128, 700, 152 * 128 * 2 + 77])
def test_tensor_core_forward(S, arm, E):
    """The tcgen05 inference (fused, tiles of 128 edges, several tiles per
    CTA for the largest E) against the FP64 reference with the same bf16
    rounding points, and against the mma.sync forward."""
    mlp = S.MLP(max_batch=4096)
    ps = seeded_params(11)
    load(mlp, ps)
    s0, s1 = synth.random_edges(arm, E, 12)
    d0, d1 = dev(s0), dev(s1)
    Y = mlp.predict(arm, d0, d1).cpu().numpy()
    assert mlp.error() == 0
    Yr = mlp.predict_ref(arm, d0, d1).cpu().numpy()
    ref, _ = M.forward([(W.astype(np.float64), b.astype(np.float64)) for W, b in ps],
                       M.features(arm, s0, s1))
    assert relerr(Y, ref) < 1e-3, relerr(Y, ref)
    ok, worst = elementwise_ok(Y, ref)
    assert ok, worst
    assert relerr(Y, Yr) < 1e-3, relerr(Y, Yr)
    # per edge: the two GPU paths differ only by FP32 summation order (and
    # the bf16 roundings that order can flip)
    assert np.abs(Y - Yr).max() <= 1e-2 * max(1.0, np.abs(Yr).max())
    mlp.close()


def test_tensor_core_forward_after_update(S, arm):
    """Weights changed by an Adam step are repacked before the next
    inference."""
    mlp = S.MLP(max_batch=512)
    load(mlp, seeded_params(13))
    s0, s1 = synth.random_edges(arm, 300, 14)
    d0, d1 = dev(s0), dev(s1)
    mlp.predict(arm, d0, d1)
    rng = np.random.default_rng(15)
    for l in range(4):
        W, b = mlp.get_params(l)
        mlp.set_grads(l, rng.normal(0, 1, W.shape).astype(np.float32),
                      rng.normal(0, 1, b.shape).astype(np.float32))
    mlp.adam_step(1e-2)
    Y = mlp.predict(arm, d0, d1).cpu().numpy()
    Yr = mlp.predict_ref(arm, d0, d1).cpu().numpy()
    assert relerr(Y, Yr) < 1e-3
    assert mlp.error() == 0
    mlp.close()


def test_gradient_parity(S, orc, arm):
    """Gradients of one batch (labels from the oracle's exact scan) agree
    norm-wise per tensor within 1e-3."""
    mlp = S.MLP(max_batch=512)
    ps = seeded_params(1)
    load(mlp, ps)
    s0, s1 = synth.random_edges(arm, 384, 4)
    grid = synth.duration_grid(32)
    lab = orc.time_edges(arm, s0, s1, grid, 8)["k_star"]
    loss = mlp.backward(arm, dev(s0), dev(s1), dev(lab.astype(np.int32)), grid)
    P64 = [(W.astype(np.float64), b.astype(np.float64)) for W, b in ps]
    y, cache = M.forward(P64, M.features(arm, s0, s1))
    feas = lab >= 0
    logT = np.log(grid.astype(np.float64))[np.clip(lab, 0, None)]
    L, dy = M.loss_and_grad_y(y, logT, feas)
    grads = M.backward(P64, cache, dy)
    assert loss == pytest.approx(L, rel=1e-3)
    for l in range(4):
        gW, gb = mlp.get_grads(l)
        assert relerr(gW, grads[l][0]) < 1e-3, (l, relerr(gW, grads[l][0]))
        assert relerr(gb, grads[l][1]) < 1e-3, (l, relerr(gb, grads[l][1]))
    mlp.close()


@pytest.mark.parametrize("E", [1, 63, 64, 65, 128, 129, 513, 152 * 128 + 77])
def test_gradient_of_ragged_batches(S, arm, E):
    """One row, the edges of the 64-row blocks, 128-row tiles and 512-row
    stages, and more tiles than SMs, in a workspace of exactly E rows, with
    feasible and infeasible labels: norm-wise within 1e-3 of the FP64 reference
    with the same rounding points (a rounding that falls the other way moves a
    tensor by up to 2^-9 / sqrt(E)); a second call gives the same again."""
    mlp = S.MLP(max_batch=E)
    ps = seeded_params(21)
    load(mlp, ps)
    s0, s1 = synth.random_edges(arm, E, 22)
    grid = synth.duration_grid(48)
    lab = np.random.default_rng(23).integers(-1, 48, E).astype(np.int32)
    lab[0] = 7
    P64 = [(W.astype(np.float64), b.astype(np.float64)) for W, b in ps]
    y, cache = M.forward(P64, M.features(arm, s0, s1))
    logT = np.log(grid.astype(np.float64))[np.clip(lab, 0, None)]
    L, dy = M.loss_and_grad_y(y, logT, lab >= 0)
    grads = M.backward(P64, cache, dy)
    for _ in range(2):
        loss = mlp.backward(arm, dev(s0), dev(s1), dev(lab), grid)
        assert mlp.error() == 0
        assert loss == pytest.approx(L, rel=1e-3)
        for l in range(4):
            gW, gb = mlp.get_grads(l)
            tol = max(1e-3, 2.0 ** -9 / np.sqrt(E))
            assert relerr(gW, grads[l][0]) < tol and relerr(gb, grads[l][1]) < tol, l
    mlp.close()


def test_adam_step_parity(S, arm):
    mlp = S.MLP(max_batch=64)
    ps = seeded_params(2)
    load(mlp, ps)
    rng = np.random.default_rng(3)
    grads = [(rng.normal(0, 1, W.shape).astype(np.float32), rng.normal(0, 1, b.shape).astype(np.float32))
             for W, b in ps]
    for l, (gW, gb) in enumerate(grads):
        mlp.set_grads(l, gW, gb)
    m = [(np.zeros(W.shape), np.zeros(b.shape)) for W, b in ps]
    P64 = [(W.astype(np.float64), b.astype(np.float64)) for W, b in ps]
    G64 = [(gW.astype(np.float64), gb.astype(np.float64)) for gW, gb in grads]
    ref, _, _ = M.adam(P64, G64, m, m, 1, 1e-3)
    mlp.adam_step(1e-3)
    for l in range(4):
        W, b = mlp.get_params(l)
        assert relerr(W, ref[l][0]) < 1e-5 and relerr(b, ref[l][1]) < 1e-5
        assert np.allclose(W, ref[l][0], rtol=1e-5, atol=1e-7)
    mlp.close()


def test_save_load_roundtrip(S, tmp_path, arm):
    a = S.MLP(max_batch=64, seed=5)
    b = S.MLP(max_batch=64, seed=6)
    a.save(tmp_path / "w.bin")
    b.load(tmp_path / "w.bin")
    for l in range(4):
        Wa, ba = a.get_params(l)
        Wb, bb = b.get_params(l)
        assert np.array_equal(Wa, Wb) and np.array_equal(ba, bb)
    a.close(); b.close()


def test_window_scan_matches_full_scan(S, arm):
    """With any prediction the windowed scan returns the full scan's k*,
    except where the certificate relied on monotone limits and the full
    scan shows an earlier isolated feasible duration."""
    from paper_2609_22608_gb300 import ops
    E, K, Sc = 3000, 128, 32
    s0, s1 = synth.random_edges(arm, E, 8)
    d0, d1 = dev(s0), dev(s1)
    grid = synth.duration_grid(K)
    full = ops.time_edges(arm, d0, d1, grid, Sc)
    kf = full["k_star"].cpu().numpy()
    rng = np.random.default_rng(9)
    # predictions: exact, shifted, random and "infeasible" centres
    lg = np.log(grid.astype(np.float64))
    y0 = np.where(kf >= 0, lg[np.clip(kf, 0, None)], 0.0)
    Y = np.stack([y0 + rng.choice([0, 0, 0.3, -0.3, 2.0, -2.0], E), rng.choice([1.0, 1.0, -1.0], E)], 1)
    w = S.time_edges_window(arm, d0, d1, grid, Sc, dev(Y.astype(np.float32)), W=16)
    kw = w["k_star"].cpu().numpy()
    path = w["path"].cpu().numpy()
    assert set(np.unique(path)) <= {0, 1}
    fb = path == 1
    assert np.array_equal(kw[fb], kf[fb]), "fallback scans must be exact"
    mism = np.nonzero(kw != kf)[0]
    assert len(mism) <= 0.01 * E, len(mism)
    # a certified disagreement may only pick a later duration (a feasible
    # index below the certificate was missed), never an infeasible one
    Tw = w["T_star"].cpu().numpy()
    for e in mism:
        assert kw[e] == -1 or kf[e] == -1 or kw[e] > kf[e]
    okw = w["ok"].cpu().numpy()
    same = kw == kf
    assert np.array_equal(okw[same], full["ok"].cpu().numpy()[same])
    assert np.array_equal(Tw[same & (kw >= 0)], grid[kw[same & (kw >= 0)]])


def test_training_reduces_loss_and_window_hits(S, arm):
    """A short training run on edges labelled by the exact scan lowers the
    loss, and the trained network's windows certify most edges."""
    from paper_2609_22608_gb300 import ops
    E, K, Sc = 32768, 128, 32
    s0, s1 = synth.random_edges(arm, E, 10)
    d0, d1 = dev(s0), dev(s1)
    grid = synth.duration_grid(K)
    lab = S.label_edges(arm, d0, d1, grid, Sc)
    mlp = S.MLP(max_batch=4096, seed=0)
    hist = S.train(mlp, arm, d0, d1, lab, grid, epochs=3, batch=4096, lr=2e-3)
    assert hist[-1] < 0.7 * hist[0], hist
    t0, t1 = synth.random_edges(arm, 4096, 11)
    e0, e1 = dev(t0), dev(t1)
    Y = mlp.predict(arm, e0, e1)
    w = S.time_edges_window(arm, e0, e1, grid, Sc, Y, W=16)
    full = ops.time_edges(arm, e0, e1, grid, Sc)
    hit = (w["path"] == 0).float().mean().item()
    agree = (w["k_star"] == full["k_star"]).float().mean().item()
    assert hit > 0.3, hit
    assert agree > 0.99, agree
    mlp.close()


def test_trained_window_saves_work(S, arm):
    """What training buys, and what the window saves against the exact scan:
    on the same edges, with identical chosen durations, the trained
    network's window pass needs fewer torque evaluations than the window of
    an untrained network (whose misses fall back to the full scan), and
    fewer than the full scan: the window's scan starts a few grid steps
    below the predicted index, so the interior probes of the end-sample
    survivors far below k* (a pass per eight of them in the full scan) are
    skipped."""
    import torch
    from paper_2609_22608_gb300 import ops
    E, K, Sc = 32768, 128, 32
    s0, s1 = synth.random_edges(arm, E, 20)
    d0, d1 = dev(s0), dev(s1)
    grid = synth.duration_grid(K)
    lab = S.label_edges(arm, d0, d1, grid, Sc)
    trained = S.MLP(max_batch=4096, seed=0)
    S.train(trained, arm, d0, d1, lab, grid, epochs=12, batch=2048, lr=2e-3)
    untrained = S.MLP(max_batch=4096, seed=0)
    t0, t1 = synth.random_edges(arm, 4096, 21)
    e0, e1 = dev(t0), dev(t1)

    def evaluations(fn):
        c = torch.zeros(1, dtype=torch.int64, device="cuda")
        out = fn(c)
        torch.cuda.synchronize()
        return int(c.item()), out

    n_full, full = evaluations(lambda c: ops.time_edges(arm, e0, e1, grid, Sc, sample_count=c))
    n_tr, w_tr = evaluations(lambda c: S.time_edges_window(
        arm, e0, e1, grid, Sc, trained.predict(arm, e0, e1), W=16, sample_count=c))
    n_un, w_un = evaluations(lambda c: S.time_edges_window(
        arm, e0, e1, grid, Sc, untrained.predict(arm, e0, e1), W=16, sample_count=c))
    trained.close()
    untrained.close()
    assert (w_tr["k_star"] == full["k_star"]).float().mean().item() > 0.99
    assert (w_un["k_star"] == full["k_star"]).float().mean().item() > 0.99
    assert n_tr < n_un, (n_tr, n_un)
    assert n_tr < n_full, (n_tr, n_full)


def _call(fn, *args):
    import ctypes as C
    return fn(*[C.c_void_p(a.data_ptr()) if torch.is_tensor(a) else a for a in args])


@pytest.mark.parametrize("change", ["create", "set_params", "adam"])
def test_weights_packed_for_every_stream(S, arm, change):
    """After a change of the weights, a gradient queued on one busy stream (the
    loss not asked for) and a prediction on another at the same time: both see
    the new weights, whatever the first one has not come to yet."""
    import ctypes as C
    E, grid = 300, synth.duration_grid(16)
    s0, s1 = synth.random_edges(arm, E, 31)
    d0, d1 = dev(s0), dev(s1)
    lab = dev(np.random.default_rng(32).integers(-1, 16, E).astype(np.int32))
    from paper_2609_22608_gb300._lib import arm_struct, lib
    mlp = S.MLP(max_batch=512, seed=4)
    if change == "set_params":
        load(mlp, seeded_params(33))
    elif change == "adam":
        mlp.backward(arm, d0, d1, lab, grid)
        mlp.adam_step(1e-2)
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(a):
        torch.cuda._sleep(2_000_000)
    A = arm_struct(arm)
    assert _call(lib().fn_mlp_backward, mlp.h, C.byref(A), d0, d1, lab,
                 grid.ctypes.data_as(C.c_void_p), 16, E, None, C.c_void_p(a.cuda_stream)) == 0
    with torch.cuda.stream(b):
        Y = mlp.predict(arm, d0, d1, stream=b)
    torch.cuda.synchronize()
    Yr = mlp.predict_ref(arm, d0, d1).cpu().numpy()
    assert relerr(Y.cpu().numpy(), Yr) < 1e-3     # the two forwards' tolerance, as above
    mlp.close()


def test_wait_that_runs_out(S, arm):
    """Kernels that give up at their first wait, with the copies of the weights
    in flight: they raise the flag and end cleanly, and with the usual limit the
    same model gives the same results as before."""
    E, grid = 152 * 128 + 77, synth.duration_grid(16)
    s0, s1 = synth.random_edges(arm, E, 41)
    d0, d1 = dev(s0), dev(s1)
    lab = dev(np.random.default_rng(42).integers(-1, 16, E).astype(np.int32))
    mlp = S.MLP(max_batch=E)
    load(mlp, seeded_params(43))
    Y = mlp.predict(arm, d0, d1)
    mlp.backward(arm, d0, d1, lab, grid)
    g = [mlp.get_grads(l) for l in range(4)]
    assert mlp.error() == 0
    for call in ("predict", "backward"):
        mlp.set_wait(-1)
        if call == "predict":
            mlp.predict(arm, d0, d1)
        else:
            _call_backward(mlp, arm, d0, d1, lab, grid)
        torch.cuda.synchronize()
        assert mlp.error(reset=True) == 1
        mlp.set_wait(2_000_000_000)
        assert torch.equal(mlp.predict(arm, d0, d1), Y)
        mlp.backward(arm, d0, d1, lab, grid)
        assert mlp.error() == 0
        for l in range(4):           # sums in another order: FP32's 2^-24 on 2e4 rows
            for a, b in zip(mlp.get_grads(l), g[l]):
                assert relerr(a, b) < 1e-5
    mlp.close()


def _call_backward(mlp, arm, d0, d1, lab, grid):
    """fn_mlp_backward without the loss: its status."""
    import ctypes as C

    from paper_2609_22608_gb300._lib import arm_struct, lib
    A = arm_struct(arm)
    return _call(lib().fn_mlp_backward, mlp.h, C.byref(A), d0, d1, lab,
                 grid.ctypes.data_as(C.c_void_p), len(grid), d0.shape[0], None,
                 C.c_void_p(torch.cuda.current_stream().cuda_stream))


def test_gradient_given_up(S, arm):
    """A gradient whose wait ran out is reported where its loss is read and is
    never applied; the caller's own gradients and the next backward are."""
    from paper_2609_22608_gb300._lib import FnError
    E, grid = 500, synth.duration_grid(16)
    s0, s1 = synth.random_edges(arm, E, 51)
    d0, d1 = dev(s0), dev(s1)
    lab = dev(np.random.default_rng(52).integers(-1, 16, E).astype(np.int32))
    mlp = S.MLP(max_batch=E)
    load(mlp, seeded_params(53))
    mlp.backward(arm, d0, d1, lab, grid)          # images of an earlier batch
    before = [mlp.get_params(l) for l in range(4)]

    def unchanged():
        return all(np.array_equal(x, y) for l in range(4)
                   for x, y in zip(mlp.get_params(l), before[l]))
    mlp.set_wait(-1)
    with pytest.raises(FnError):
        mlp.backward(arm, d0, d1, lab, grid)
    mlp.adam_step(1e-2)
    assert unchanged()
    assert _call_backward(mlp, arm, d0, d1, lab, grid) == 0     # nothing read back
    mlp.adam_step(1e-2)
    assert unchanged()
    with pytest.raises(FnError):
        mlp.train_step(arm, d0, d1, lab, grid, 1e-2)
    assert unchanged() and mlp.error(reset=True) == 1
    for l in range(4):
        W, b = mlp.get_params(l)
        mlp.set_grads(l, np.ones_like(W), np.ones_like(b))
    mlp.adam_step(1e-2)
    assert not unchanged()
    mlp.set_wait(2_000_000_000)
    after = [mlp.get_params(l)[0] for l in range(4)]
    assert np.isfinite(mlp.train_step(arm, d0, d1, lab, grid, 1e-2)) and mlp.error() == 0
    assert not np.array_equal(mlp.get_params(1)[0], after[1])
    mlp.close()


def test_gradient_sum_of_many_rows(S, arm):
    """2^17 equal rows: every term of the first layer's weight gradient is the same
    and scales exactly with the batch, so the sum is that of 128 rows but for what
    the additions lose.  A chain on the tensor core loses at most 2^-23 a step of 16
    rows (it need not round to nearest): 76 steps to each of 4 x 27 accumulators,
    then 31 FP32 additions."""
    E, grid = 1 << 17, synth.duration_grid(16)
    s0, s1 = synth.random_edges(arm, 1, 5)
    mlp = S.MLP(max_batch=E)
    load(mlp, seeded_params(61))
    g = []
    for n in (128, E):
        mlp.backward(arm, dev(np.repeat(s0, n, 0)), dev(np.repeat(s1, n, 0)),
                     torch.full((n,), 7, dtype=torch.int32, device="cuda"), grid)
        g.append(mlp.get_grads(0)[0].astype(np.float64))
    mlp.close()
    some = g[0] != 0
    assert some.any() and np.array_equal(g[1] != 0, some)
    assert np.abs(g[1][some] / g[0][some] - 1).max() < 76 * 2.0 ** -23 + 31 * 2.0 ** -24
