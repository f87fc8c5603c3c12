"""The workspace that apsp_predecessors asks for stays bounded for float32: a caller who allocates it keeps
the sizes that worked when it was 256 bytes."""
import torch

import paper_2310_03983_gb300 as apsp


def test_float_scratch_is_bounded():
    for n in (1, 127, 128, 3000, 8192, 8193, 8200, 9000, 16400, 20000, 32768, 46341, 100000, 150000, 1 << 20, (1 << 20) + 1):
        assert 256 <= apsp.apsp_predecessors_workspace_bytes(n, torch.float32) <= 256 + (1 << 30)
    assert apsp.apsp_predecessors_workspace_bytes(8192, torch.float32) == 256 + 16 * 8192 ** 2
