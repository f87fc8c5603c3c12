"""Repeated squaring where its products change route: one launch on 64 x 64 tiles, or a loop of
products on 128 x 128 tiles, whichever is faster for the size, and for int32 up to n = 4096 packed
16-bit pairs first.  Which one runs shows in the launch count; the results equal the oracle's (int32
exactly, float32 within 1e-5 relative)."""
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


def _products(n):
    return max(0, int(np.ceil(np.log2(n - 1))))


# On 152 SMs 1448, 2048, 3072 and 4096 need more rounds of 64 x 64 tiles than they are worth; 1024 and
# 2896 do not.  int32 starts with the 16-bit products and keeps the tiles up to 2048 all the same.
@pytest.mark.parametrize("n", [1024, 1448, 2048, 2896, 3072, 4096, 4097])
@pytest.mark.parametrize("dtype", ["int32", "float32"])
def test_launches_and_sampled_rows(apsp, n, dtype):
    loop = n in ((1448, 2048, 3072, 4096, 4097) if dtype == "float32" else (3072, 4096, 4097))
    kw = {"lo": 1, "hi": 100} if dtype == "int32" else {"dist": "lognormal", "lo": 0.0, "hi": 1.0}
    h = workloads.er_graph(n, 0.02, dtype, seed=n, **kw)
    d = torch.from_numpy(h).cuda()
    apsp.apsp_launch_count(reset=True)
    apsp.apsp_squaring(d)
    got = apsp.apsp_launch_count()
    packed = dtype == "int32" and n <= 4096
    ld_copies = 2 if n % 4 else 0
    # a1 (packed: a1 with the packing, the 16-bit products, their result), then the 32-bit products
    assert got == ld_copies + (3 if packed else 1) + (2 * _products(n) if loop else 2)
    assert apsp.apsp_device_status() == 0
    rows = np.sort(np.random.default_rng(n).choice(n, 24, replace=False))
    assert_dist_equal(d.cpu().numpy()[rows], oracle.dijkstra_rows(h, rows, threads=THREADS), f"squaring n={n} {dtype}")


@pytest.mark.parametrize("w", [1, 6, 40, 9000])
@pytest.mark.parametrize("iters", [1, 2, 10, 11, 48])
def test_path_by_products_in_the_loop(apsp, w, iters):
    """A path of 2499 edges of weight w: t products reach the pairs up to 2^t apart.  w = 1 stays on 16-bit
    pairs, w = 6 outgrows them in the last products, w = 40 earlier, w = 9000 starts beyond them: the
    loop has to go on where they stopped, by as many products as are left."""
    n = 2500
    h = np.full((n, n), INF, np.int32)
    np.fill_diagonal(h, 0)
    h[np.arange(n - 1), np.arange(1, n)] = w
    gap = np.arange(n, dtype=np.int32)[None, :] - np.arange(n, dtype=np.int32)[:, None]
    want = np.where((gap >= 0) & (gap <= 2 ** iters), gap * w, INF)
    base = apsp.apsp_squaring_workspace_bytes(n, n, torch.float32)  # no room for the packed operands
    for ws in (None, torch.empty(base, dtype=torch.uint8, device="cuda")):
        d = torch.from_numpy(h).cuda()
        apsp.apsp_launch_count(reset=True)
        apsp.apsp_squaring(d, max_iters=iters, ws=ws)
        assert apsp.apsp_launch_count() == (3 if ws is None else 1) + 2 * min(iters, 12)
        assert np.array_equal(d.cpu().numpy(), want)
    assert apsp.apsp_device_status() == 0


def test_loop_after_16_bit_products_in_a_graph(apsp):
    """Captured once, replayed on other weights: the skip words are set anew by each replay."""
    n = 2500
    ws = torch.empty(apsp.apsp_squaring_workspace_bytes(n, n), dtype=torch.uint8, device="cuda")
    hs = [workloads.er_graph(n, 0.005, "int32", lo=1, hi=hi, seed=hi) for hi in (100, 10**5, 4000, 100)]
    d = torch.from_numpy(hs[0]).cuda()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        apsp.apsp_squaring(d, ws=ws)  # per-device set-up before capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        apsp.apsp_squaring(d, ws=ws)
    for h in hs:
        d.copy_(torch.from_numpy(h).cuda())
        want = d.clone()
        apsp.apsp_fw(want)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(d, want)
    assert apsp.apsp_device_status() == 0
