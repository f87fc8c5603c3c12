"""Products on 64 x 64 tiles whose tiles outnumber the consumer groups (304 on 152 SMs), so that every group
takes several: the operand ring and the old tile's barrier carried from tile to tile, folded into C or
not, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_parity import assert_dist_equal

pytestmark = pytest.mark.gpu
INF = workloads.INF_I32


@pytest.fixture(scope="module")
def apsp():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2310_03983_gb300 as m
    assert m.apsp_device_status() == 0
    return m


# 812 tiles (the last row and column partial) at one and two chunks of k, 1100 tiles, 2 x 2000 tiles.
@pytest.mark.parametrize("m,n,k", [(1790, 1800, 64), (1790, 1800, 70), (1590, 2810, 33), (130, 128000, 20)])
@pytest.mark.parametrize("kind", ["int32", "heavy", "f32"])
def test_products(apsp, m, n, k, kind):
    rng = np.random.default_rng(m + n + k)
    dt = np.float32 if kind == "f32" else np.int32
    none = np.inf if kind == "f32" else INF

    def mat(r, c):
        v = rng.lognormal(0, 1, (r, c)) if kind == "f32" else rng.integers(1, 10**6 if kind == "heavy" else 100, (r, c))
        x = np.where(rng.random((r, c)) < 0.6, v, none).astype(dt)
        t = torch.zeros((r, (c + 3) // 4 * 4), dtype=torch.float32 if kind == "f32" else torch.int32, device="cuda")
        t[:, :c] = torch.from_numpy(x).cuda()
        return x, t[:, :c]

    (a, A), (b, B), (c, C) = mat(m, k), mat(k, n), mat(m, n)
    for acc in (True, False):
        out = torch.empty((m, (n + 3) // 4 * 4), dtype=C.dtype, device="cuda")[:, :n]
        out.copy_(C)
        apsp.tropical_gemm(out, A, B, accumulate=acc)
        want = oracle.minplus(a, b)
        want = np.minimum(want, c) if acc else want
        assert_dist_equal(out.cpu().numpy(), want.astype(dt) if dt == np.int32 else want, f"{m}x{n}x{k} {kind}")
    assert apsp.apsp_device_status() == 0
