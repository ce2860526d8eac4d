"""Parity of the CUDA nearest-parent search (fn_knn_tree) with the oracle's
brute force."""
import numpy as np
import pytest
import torch

from paper_2609_22608_gb300 import synth
from tests.parity import knn_mismatches

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ops():
    from paper_2609_22608_gb300 import ops as o
    return o


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("B,N,k,first,ws", [
    (2048, 4096, 8, 1, True),     # planning-iteration shape
    (2048, 4096, 8, 1, False),    # single-pass path (no workspace)
    (300, 1000, 16, 1, True),
    (129, 257, 5, 0, True),
    (7, 3, 4, 1, True),           # fewer candidates than k
    (1, 1, 1, 1, True),           # only the root: nothing to return
    (64, 130, 16, 0, False),
])
def test_knn_parity(ops, orc, arm, B, N, k, first, ws):
    tree = synth.random_states(arm, N, 5 + N)
    q = synth.random_states(arm, B, 6 + B)
    if N > 20:
        tree[N // 2] = tree[3]          # exact duplicates: ties go to the lower index
        q[0] = tree[3]
    workspace = None
    if ws:
        need = ops.knn_workspace_bytes(B, N, k)
        workspace = torch.empty(max(need, 1) + 256, dtype=torch.uint8, device="cuda")
    idx, d2 = ops.knn_tree(dev(tree), dev(q), k, 0.1, first=first, workspace=workspace)
    ig, dg = idx.cpu().numpy(), d2.cpu().numpy()
    ri, rd = orc.knn(tree, q, k, 0.1, first=first)
    bad = knn_mismatches(ig, dg, ri, rd)
    assert not bad, (bad[:4], ig[bad[0]], ri[bad[0]])
    fin = np.isfinite(rd)
    assert np.allclose(dg[fin], rd[fin], rtol=1e-5, atol=1e-6)
    assert np.all(ig[~fin] == -1)
    if N > 20 and first <= 3:
        assert ig[0, 0] == 3 and ig[0, 1] == N // 2


def test_knn_full_size_sampled(ops, orc, arm):
    """The anytime-stress shape (8192 queries, 65536 nodes, k = 16): sampled
    queries against the brute force, and sortedness everywhere."""
    B, N, k = 8192, 65536, 16
    tree = synth.random_states(arm, N, 99)
    q = synth.random_states(arm, B, 98)
    idx, d2 = ops.knn_tree(dev(tree), dev(q), k, 0.1)
    ig, dg = idx.cpu().numpy(), d2.cpu().numpy()
    assert np.all(np.diff(dg, axis=1) >= 0)
    sel = np.random.default_rng(1).choice(B, 64, replace=False)
    ri, rd = orc.knn(tree, q[sel], k, 0.1)
    assert not knn_mismatches(ig[sel], dg[sel], ri, rd)


def _scan(tree, q, k, first, w=0.1):
    """fn_knn_tree without a workspace: the FP32 scan of every node."""
    import ctypes as C

    from paper_2609_22608_gb300._lib import lib
    B = q.shape[0]
    idx = torch.empty(B, k, dtype=torch.int32, device="cuda")
    d2 = torch.empty(B, k, device="cuda")
    st = lib().fn_knn_tree(C.c_void_p(tree.data_ptr()), tree.shape[0], first,
                           C.c_void_p(q.data_ptr()), B, k, w, C.c_void_p(idx.data_ptr()),
                           C.c_void_p(d2.data_ptr()), None, 0,
                           C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    return idx, d2


def _odd_states(kind, arm, N, B):
    t, q = synth.random_states(arm, N, N), synth.random_states(arm, B, N + B)
    rng = np.random.default_rng(N)
    if kind == "copies":                      # ties everywhere
        t = t[rng.integers(0, 9, N)]
        q[::2] = t[rng.integers(0, N, len(q[::2]))]
    elif kind == "tight":                     # clusters below the filter's resolution
        t = t[rng.integers(0, 4, N)] + 1e-4 * rng.standard_normal((N, 16)).astype(np.float32)
        q[:] = t[rng.integers(0, N, B)]
    elif kind == "tiny":
        t, q = t * np.float32(1e-4), q * np.float32(1e-4)
    elif kind == "outside":                   # states the filter's operands cannot hold
        t[5, 3], t[17, 0], t[40], t[N - 1, 9] = np.nan, np.inf, 1e20, -np.inf
        t[60] *= 60
        q[0, 2], q[1], q[2, 1] = np.nan, 1e20, np.inf
        q[3], q[4] = t[40], q[4] * 1000
    elif kind == "few":                       # fewer finite nodes than k
        t[7:] = np.inf
    return t.astype(np.float32), q.astype(np.float32)


@pytest.mark.parametrize("kind", ["uniform", "copies", "tight", "tiny", "outside", "few"])
@pytest.mark.parametrize("B,N,k,first", [(5, 257, 1, 1), (256, 384, 8, 0), (257, 2049, 16, 1),
                                         (64, 4000, 7, 100), (700, 8320, 9, 1)])
def test_knn_filter_is_the_scan(ops, arm, kind, B, N, k, first):
    """The tensor-core filter's lists are the FP32 scan's bit for bit: sizes at
    the edges of its groups, tiles and row blocks, and states where its scores
    tie, coincide or do not exist."""
    t, q = (dev(x) for x in _odd_states(kind, arm, N, B))
    ws = torch.full((ops.knn_workspace_bytes(B, N, k) + 256,), 0xFF, dtype=torch.uint8,
                    device="cuda")            # contents on entry do not matter (NaNs here)
    idx, d2 = ops.knn_tree(t, q, k, 0.1, first=first, workspace=ws)
    ri, rd = _scan(t, q, k, first)
    assert torch.equal(idx, ri)
    assert torch.equal(d2.view(torch.int32), rd.view(torch.int32))


def test_knn_on_side_streams(ops, arm):
    """Searches queued on two busy side streams, their workspaces left to the
    call: what the current stream and the other side stream allocate and write
    meanwhile must not be theirs."""
    B, N, k = 300, 700, 8                     # a tree that the filter takes
    t = [dev(synth.random_states(arm, N, 70 + i)) for i in range(2)]
    q = [dev(synth.random_states(arm, B, 80 + i)) for i in range(2)]
    ref = [_scan(t[i], q[i], k, 1) for i in range(2)]
    need = ops.knn_workspace_bytes(B, N, k)
    assert need > 0
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for _ in range(4):
        for i, s in enumerate(streams):
            with torch.cuda.stream(s):
                torch.cuda._sleep(1_000_000)  # the search waits; the host goes on
            got.append((i, ops.knn_tree(t[i], q[i], k, 0.1, stream=s)))
            torch.full((need + 256,), 0xFF, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    for i, (idx, d2) in got:
        assert torch.equal(idx, ref[i][0])
        assert torch.equal(d2.view(torch.int32), ref[i][1].view(torch.int32))


@pytest.mark.parametrize("kind", ["same", "tight", "degrees", "one_out"])
@pytest.mark.parametrize("B,N,k", [(1, 20003, 8), (3, 4099, 16), (130, 9000, 5), (2500, 1030, 16),
                                   (5003, 2100, 8)])
def test_knn_without_help_of_the_filter(ops, arm, kind, B, N, k):
    """Queries whose scores tell nothing apart (eight to one warps each): coinciding
    nodes, clusters below the scores' error, states outside their range, and one
    such query among ordinary ones.  The scan's lists bit for bit."""
    t, q = synth.random_states(arm, N, N), synth.random_states(arm, B, N + B)
    rng = np.random.default_rng(N)
    if kind == "same":
        t[:] = t[0]
    elif kind == "tight":
        t = t[rng.integers(0, 4, N)] + 1e-4 * rng.standard_normal((N, 16)).astype(np.float32)
        q[::2] = t[rng.integers(0, N, len(q[::2]))]
    elif kind == "degrees":
        t, q = t * np.float32(57.3), q * np.float32(57.3)
    else:
        q[B // 2] *= 1000
    t, q = dev(t.astype(np.float32)), dev(q.astype(np.float32))
    idx, d2 = ops.knn_tree(t, q, k, 0.1)
    ri, rd = _scan(t, q, k, 1)
    assert torch.equal(idx, ri)
    assert torch.equal(d2.view(torch.int32), rd.view(torch.int32))


@pytest.mark.parametrize("w", [0.0, 1e-20, 1.0, 80.0, 3e3, 1e4, 1e30, 3e38])
def test_knn_velocity_weights(ops, arm, w):
    """Weights that need the filter's operands scaled, up to FP32's largest: the
    scan's lists bit for bit."""
    t, q = dev(synth.random_states(arm, 5000, 3)), dev(synth.random_states(arm, 333, 4))
    idx, d2 = ops.knn_tree(t, q, 9, w)
    ri, rd = _scan(t, q, 9, 1, w)
    assert torch.equal(idx, ri)
    assert torch.equal(d2.view(torch.int32), rd.view(torch.int32))


@pytest.mark.parametrize("tiles", [0, 1, 2, 5])
def test_knn_in_a_smaller_workspace(ops, arm, tiles):
    """A workspace that holds the nodes and only some tiles of 256 queries: the same
    lists in more batches; with no tile, the scan's split pass."""
    B, N, k = 1500, 3000, 6
    t, q = dev(synth.random_states(arm, N, 5)), dev(synth.random_states(arm, B, 6))
    ri, rd = _scan(t, q, k, 1)
    one, two = (ops.knn_workspace_bytes(b, N, k) for b in (256, 512))
    size = one + (tiles - 1) * (two - one) if tiles else one - 256
    ws = torch.full((size + 256 + 1024,), 0x7F, dtype=torch.uint8, device="cuda")
    off = -ws.data_ptr() % 256
    idx, d2 = ops.knn_tree(t, q, k, 0.1, workspace=ws[off:off + size])
    assert torch.equal(idx, ri)
    assert torch.equal(d2.view(torch.int32), rd.view(torch.int32))
    assert (ws[off + size:] == 0x7F).all()


@pytest.mark.parametrize("N,B,rows,filtered", [
    (257, 40000, 13568, True), (257, 40000, 10240, False),       # 3 batches pay, 4 do not
    (700, 40000, 5888, True), (700, 40000, 5632, False)])        # 7 and 8
def test_knn_batches_that_pay(ops, arm, N, B, rows, filtered):
    """A workspace of `rows` queries serves the filter while the batches are few, and is
    left alone where the scan in one launch is faster.  The same lists either way."""
    k = 4
    t, q = dev(synth.random_states(arm, N, 7)), dev(synth.random_states(arm, B, 8))
    ri, rd = _scan(t, q, k, 1)
    one, two = (ops.knn_workspace_bytes(b, N, k) for b in (32768, 33024))
    size = one + (rows - 32768) // 256 * (two - one)
    ws = torch.full((size + 256,), 0x7F, dtype=torch.uint8, device="cuda")
    off = -ws.data_ptr() % 256
    idx, d2 = ops.knn_tree(t, q, k, 0.1, workspace=ws[off:off + size])
    assert torch.equal(idx, ri)
    assert torch.equal(d2.view(torch.int32), rd.view(torch.int32))
    assert bool((ws != 0x7F).any()) == filtered
