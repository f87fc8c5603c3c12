"""The kernels on 64 x 64 tiles against the oracle, at the edges of their tiles and ranges: the closure of
small matrices, small products and repeated squaring.  int32 is bit-exact; float32 is within 1e-5
relative of fp64 (a path of L edges is off by at most (L - 1) 2^-24)."""
import os

import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_parity import assert_dist_equal

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 4
INF = workloads.INF_I32


@pytest.fixture(scope="module")
def apsp():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2310_03983_gb300 as m
    assert m.apsp_device_status() == 0
    return m


def _graph(n, kind, seed):
    p = 0.05 if n > 100 else 0.3
    if kind == "f32":
        return workloads.er_graph(n, p, "float32", dist="lognormal", lo=0.0, hi=1.0, seed=seed)
    return workloads.er_graph(n, p, "int32", lo=1, hi=10**6 if kind == "heavy" else 100, seed=seed)


def _check(apsp, d, h, what):
    assert apsp.apsp_device_status() == 0
    if h.shape[0] <= 1100:
        assert_dist_equal(d.cpu().numpy(), oracle.fw(h, threads=THREADS), what)
    else:
        rows = np.sort(np.random.default_rng(h.shape[0]).choice(h.shape[0], 24, replace=False))
        assert_dist_equal(d.cpu().numpy()[rows], oracle.dijkstra_rows(h, rows, threads=THREADS), what)


# 129 and 3200: the ends of the range; one and two groups of tiles per SM from n = 1730
@pytest.mark.parametrize("kind", ["int32", "heavy", "f32"])
@pytest.mark.parametrize("n", [129, 191, 192, 193, 254, 320, 1000, 1793, 3200])
def test_closure(apsp, n, kind):
    h = _graph(n, kind, n)
    d = torch.from_numpy(h).cuda()
    apsp.apsp_fw(d)
    _check(apsp, d, h, f"fw n={n} {kind}")


def test_closure_in_a_wider_matrix_leaves_the_rest(apsp):
    h = _graph(257, "int32", 5)
    full = torch.full((260, 384), -7, dtype=torch.int32, device="cuda")
    full[:257, :257] = torch.from_numpy(h).cuda()
    apsp.apsp_fw(full[:257, :257])
    _check(apsp, full[:257, :257], h, "fw in a view")
    assert torch.all(full[257:] == -7) and torch.all(full[:, 257:] == -7)


@pytest.mark.parametrize("kind", ["int32", "heavy", "f32"])
@pytest.mark.parametrize("n", [2, 63, 64, 65, 130, 333, 1030, 1100])
def test_squaring(apsp, n, kind):
    h = _graph(n, kind, n + 1)
    d = torch.from_numpy(h).cuda()
    apsp.apsp_squaring(d)
    _check(apsp, d, h, f"squaring n={n} {kind}")


@pytest.mark.parametrize("w", [1, 40, 9000])
@pytest.mark.parametrize("iters", [1, 2, 5, 9, 48])
def test_squaring_of_a_path_by_products(apsp, w, iters):
    """A path of 700 edges of weight w: t products reach the pairs up to 2^t apart.  w = 40 outgrows
    the 16-bit pairs on the way (the rest runs on 32 bits), w = 9000 starts beyond them."""
    n = 701
    h = np.full((n, n), INF, np.int32)
    np.fill_diagonal(h, 0)
    h[np.arange(n - 1), np.arange(1, n)] = w
    d = torch.from_numpy(h).cuda()
    apsp.apsp_squaring(d, max_iters=iters)
    gap = np.arange(n)[None, :] - np.arange(n)[:, None]
    want = np.where((gap >= 0) & (gap <= 2 ** iters), gap * w, INF)
    assert np.array_equal(d.cpu().numpy(), want)
    assert apsp.apsp_device_status() == 0


def test_squaring_without_room_for_the_packed_operands(apsp):
    h = _graph(300, "int32", 9)
    full = apsp.apsp_squaring_workspace_bytes(300, 300)
    base = apsp.apsp_squaring_workspace_bytes(300, 300, torch.float32)
    assert base < full
    for size in (base, full):
        d = torch.from_numpy(h).cuda()
        apsp.apsp_squaring(d, ws=torch.empty(size, dtype=torch.uint8, device="cuda"))
        _check(apsp, d, h, f"squaring ws={size}")


@pytest.mark.parametrize("kind", ["int32", "heavy", "f32"])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (64, 64, 64), (65, 63, 130), (200, 300, 101), (257, 1025, 511), (700, 90, 2000)])
def test_product(apsp, m, n, k, kind):
    rng = np.random.default_rng(m + n + k)
    dt = np.float32 if kind == "f32" else np.int32
    hi = 10**6 if kind == "heavy" else 100

    def mat(r, c):  # 16-byte rows, so the tiles are loaded by TMA
        v = rng.lognormal(0, 1, (r, c)) if kind == "f32" else rng.integers(1, hi + 1, (r, c))
        x = np.where(rng.random((r, c)) < 0.6, v, np.inf if kind == "f32" else INF).astype(dt)
        t = torch.zeros((r, (c + 3) // 4 * 4), dtype=torch.float32 if kind == "f32" else torch.int32, device="cuda")
        t[:, :c] = torch.from_numpy(x).cuda()
        return x, t[:, :c]

    (a, A), (b, B), (c, C) = mat(m, k), mat(k, n), mat(m, n)
    for acc in (True, False):
        out = torch.empty((m, (n + 3) // 4 * 4), dtype=C.dtype, device="cuda")[:, :n]
        out.copy_(C)
        apsp.tropical_gemm(out, A, B, accumulate=acc)
        want = oracle.minplus(a, b)
        if acc:
            want = np.minimum(want, c)
        assert_dist_equal(out.cpu().numpy(), want.astype(np.int32) if dt == np.int32 else want, f"{m}x{n}x{k} {kind}")
    assert apsp.apsp_device_status() == 0


@pytest.mark.parametrize("dtype", ["int32", "float32"])
@pytest.mark.parametrize("m,n,k", [(255, 257, 255), (301, 303, 305), (513, 511, 514), (640, 129, 1001)])
def test_product_of_unaligned_operands(apsp, m, n, k, dtype):
    """Contiguous operands whose rows are not 16-byte aligned (or only some of them): below and above the
    sizes that run on aligned copies, with and without a caller workspace, and folded into C."""
    rng = np.random.default_rng(m + k)
    dt = np.dtype(dtype)

    def mat(r, c):
        v = rng.lognormal(0, 1, (r, c)) if dtype == "float32" else rng.integers(1, 1000, (r, c))
        return np.where(rng.random((r, c)) < 0.6, v, np.inf if dtype == "float32" else INF).astype(dt)

    a, b, c = mat(m, k), mat(k, n), mat(m, n)
    A, B = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    for acc in (False, True):
        want = np.minimum(oracle.minplus(a, b), c) if acc else oracle.minplus(a, b)
        for w in (None, ws):
            out = torch.from_numpy(c).cuda()
            apsp.tropical_gemm(out, A, B, accumulate=acc, ws=w)
            assert_dist_equal(out.cpu().numpy(), want.astype(dt) if dtype == "int32" else want, f"{m}x{n}x{k} {dtype}")
    assert apsp.apsp_device_status() == 0


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("n", [127, 128, 129, 300, 513, 1001])
def test_float_predecessors(apsp, n, ties):
    """The smallest last hop, index for index, with the chunked product (from n = 128) and with the direct
    kernel (a workspace without room for the copies); ties: half-integer weights."""
    h = _graph(n, "f32", n + 3)
    if ties:
        h = np.where(np.isfinite(h), np.ceil(2 * h) / 2, h).astype(np.float32)
        np.fill_diagonal(h, 0)
    w = torch.from_numpy(h).cuda()
    d = w.clone()
    apsp.apsp_fw(d)
    want = oracle.last_hop(d.cpu().numpy(), h, threads=THREADS)
    full = apsp.apsp_predecessors_workspace_bytes(n, torch.float32)
    wide = torch.full((n, n + 5), -7, dtype=torch.int32, device="cuda")  # rows of pred not 16-byte aligned
    for ws in (None, torch.empty(256, dtype=torch.uint8, device="cuda"), torch.empty(full, dtype=torch.uint8, device="cuda")):
        apsp.apsp_predecessors(d, w, wide[:, :n], ws=ws)
        assert np.array_equal(wide[:, :n].cpu().numpy(), want)
    assert torch.all(wide[:, n:] == -7)
    assert apsp.apsp_device_status() == 0


@pytest.mark.parametrize("kind", ["int32", "heavy", "f32"])
@pytest.mark.parametrize("sizes", [[257], [384, 385, 300, 129, 256, 64], [1025, 2048, 1, 640, 200], [700] * 5])
def test_small_batch(apsp, sizes, kind):
    """Batches small enough for 64-vertex blocks in lockstep (257..2048 vertices; padding tiles skipped),
    with smaller graphs beside them on the persistent kernel (129..256: shared by a cluster)."""
    mats = [_graph(n, kind, 31 * n + g) for g, n in enumerate(sizes)]
    b = apsp.Batch(mats)
    apsp.apsp_batched(b)
    assert apsp.apsp_device_status() == 0
    out = b.pool.cpu()
    for g, m in enumerate(mats):
        _check(apsp, b.graph(g, out), m, f"graph {g} n={sizes[g]} {kind}")
