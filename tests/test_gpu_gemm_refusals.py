"""What tropical_gemm refuses does not depend on whether scratch for aligned copies may be taken."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,ok", [(64 * 65535, True), (64 * 65535 + 1, False)])
@pytest.mark.parametrize("with_ws", [False, True])
def test_rows_of_unaligned_products(rows, ok, with_ws):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2310_03983_gb300 as apsp
    a = torch.ones((rows, 5), device="cuda")  # 2^24 pairs and more: worth aligned copies
    b = torch.ones((5, 1), device="cuda")
    c = torch.zeros((rows, 1), device="cuda")
    ws = torch.empty(256, dtype=torch.uint8, device="cuda") if with_ws else None
    if ok:
        apsp.tropical_gemm(c, a, b, ws=ws)
        assert bool((c == 2).all())
    else:
        with pytest.raises(apsp.ApspError):
            apsp.tropical_gemm(c, a, b, ws=ws)
        assert bool((c == 0).all())
    assert apsp.apsp_device_status() == 0
