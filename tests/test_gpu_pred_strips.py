"""float32 predecessors by chunks where one pass of the persistent product takes many tiles per SM, and
beyond the scratch bound strip by strip, index for index against the direct kernel (which runs with a
256-byte workspace; tests/test_gpu_tiles64.py compares both with the oracle on small graphs)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def apsp():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2310_03983_gb300 as m
    assert m.apsp_device_status() == 0
    return m


# 1500: 576 tiles, two per group; 8192: the last single strip; 8200 and 9000: two strips of rows and of
# columns, unaligned rows; ties: sums of few distinct values.
@pytest.mark.parametrize("n", [1500, 3000, 8192, 8200, 9003])
@pytest.mark.parametrize("ties", [False, True])
def test_chunks_and_strips_match_the_direct_kernel(apsp, n, ties):
    g = torch.Generator(device="cuda").manual_seed(n + ties)
    d = torch.empty((n, n), device="cuda").log_normal_(0, 1, generator=g)
    w = torch.empty((n, n), device="cuda").log_normal_(0, 1, generator=g)
    if ties:
        d, w = (2 * d).ceil() / 2, (2 * w).ceil() / 2
    d.masked_fill_(torch.rand((n, n), device="cuda", generator=g) > 0.9, float("inf"))
    w.masked_fill_(torch.rand((n, n), device="cuda", generator=g) > 0.2, float("inf"))
    w[:, n // 2] = float("inf")  # a vertex no edge reaches
    d[7, :] = float("inf")       # a row that reaches nothing
    want = apsp.apsp_predecessors(d, w, ws=torch.empty(256, dtype=torch.uint8, device="cuda"))
    got = apsp.apsp_predecessors(d, w)
    assert torch.equal(got, want)
    if n > 8192:
        room = torch.empty(apsp.apsp_predecessors_workspace_bytes(n, torch.float32), dtype=torch.uint8, device="cuda")
        assert torch.equal(apsp.apsp_predecessors(d, w, ws=room), want)
    assert bool((got[:, n // 2] == -1).all()) and bool((got[7] == -1).all())
    assert apsp.apsp_device_status() == 0


def test_bad_entries_are_flagged_in_every_strip(apsp):
    n = 8300
    d = torch.ones((n, n), device="cuda")
    for which in ("d", "w"):
        for i, j in ((0, 1), (n - 1, n - 2), (n - 1, 0)):
            w, e = torch.ones((n, n), device="cuda"), d.clone()
            (e if which == "d" else w)[i, j] = -1.0
            apsp.apsp_predecessors(e, w)
            assert apsp.apsp_device_status() != 0
    apsp.apsp_predecessors(d, torch.ones((n, n), device="cuda"))
    assert apsp.apsp_device_status() == 0
