"""Epilogues of the tensor-core Legendre sums: none, two or four column blocks held per warp, by blocks per warp and by
K blocks per item.  A map alone has at most one block per warp and takes the plain loop, so that eight maps equal
their maps one by one, bit for bit, whichever epilogue runs."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu


# 8 maps of P modes: (P + 1) // 2 blocks per warp, 1 to 8.  K blocks of the longest item: 3xTF32 5, 6, 7 and 8; FP16x3 3 and 8
@pytest.mark.parametrize("prec,lmax,nphi", [("3xtf32", 158, 512), ("3xtf32", 160, 512), ("3xtf32", 222, 512), ("3xtf32", 224, 512),
                                            ("fp16x3", 160, 512), ("fp16x3", 448, 1024)])
@pytest.mark.parametrize("P", [1, 3, 4, 5, 7, 9, 11, 14, 16])
def test_epilogues_agree_bit_for_bit(prec, lmax, nphi, P):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    cl = simgen.cl_model(lmax)
    plan = M.Plan(lmax, P, simgen.shifted_legendre_basis(lmax, P), cl, lmax + 3, nphi, prec=prec)
    alm = torch.from_numpy(simgen.gaussian_alm(cl, 8, seed=P).astype(np.complex64)).cuda()
    whole = plan.synthesize(alm)
    for b in (0, 3, 7):
        assert torch.equal(whole[b], plan.synthesize(alm[b:b + 1].contiguous())[0])
    assert bool(torch.isfinite(whole).all()) and float(whole.abs().max()) > 0
    plan.sync()
    plan.close()
