"""Which channel tile the transposed FP32 Legendre sums take depends on the number of channels and of blocks; each
output is one chain of multiply-adds whatever the tile, so a batch gives each map the bits it gives alone."""
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu


# tiles of 2 (few blocks), 8, 16 and 32 channels against the 2-channel tile of a single map
@pytest.mark.parametrize("lmax,maps", [(24, 13), (128, 20), (250, 11), (128, 64)])
def test_analysis_batch_equals_single_maps(lmax, maps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    plan = M.Plan(lmax, 1, simgen.shifted_legendre_basis(lmax, 1), simgen.cl_model(lmax), lmax + 3, 512)
    plan.set_chunk(maps)
    x = torch.from_numpy(simgen.pixel_normals(lmax + 3, 512, maps, seed=5)).float().cuda()
    whole = plan.analyze(x)
    assert torch.equal(whole, torch.cat([plan.analyze(x[b:b + 1].contiguous()) for b in range(maps)]))
    plan.close()
