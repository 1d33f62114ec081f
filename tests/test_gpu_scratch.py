"""Scratch that kernel-level calls take from the library's pool goes back."""
import pytest

import paper_1704_07458_gb300 as gb
from gpu_util import torch_cuda, dev, dev_i32

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _keep(torch):
    """A call whose scratch (slab sums of the FP64 Gram) stays in the pool;
    returns the free memory before it."""
    n, p = 100000, 128
    U = torch.ones((n, p), dtype=torch.float64, device="cuda")
    G = torch.empty((p, p), dtype=torch.float64, device="cuda")
    need = gb.lobpcg_gram_workspace(n, p, p, gb.LOBPCG_GEMM_F64)
    assert 8 * MB < need <= 64 * MB
    gb.lobpcg_release_scratch()
    before = torch.cuda.mem_get_info()[0]
    assert gb.lobpcg_gram(n, U, p, p, U, p, p, G, p, gb.LOBPCG_GEMM_F64) == 0
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] <= before - need
    return before


def _chebyshev():
    c = gb.lobpcg_chebyshev_create(1, dev_i32([0, 1]), dev_i32([0]), dev([2.0]), None, 1, 0.5, 2.0,
                                   1)
    gb.lobpcg_chebyshev_destroy(c)


def _handle():
    gb.lobpcg_destroy(gb.lobpcg_create())


@pytest.mark.parametrize("give_back", [gb.lobpcg_release_scratch, _handle, _chebyshev])
def test_kept_scratch_goes_back(give_back):
    torch = torch_cuda()
    _keep(torch)  # first: kernels that load lazily, torch's own blocks
    give_back()
    before = _keep(torch)
    give_back()
    assert torch.cuda.mem_get_info()[0] >= before
