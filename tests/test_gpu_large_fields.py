"""A truncated even/odd solve whose interleaved blocks of 16 systems exceed
2^31 - 1 bytes, the largest row pitch that a two-dimensional copy or fill takes:
its vectors are then set up row by row."""
import numpy as np
import pytest
import torch

from paper_1401_6749_gb300 import synth

from .gpu_util import require_gpu

pytestmark = pytest.mark.gpu


def test_solve_beyond_two_gigabytes_per_block():
    tl = require_gpu()
    L, n = (40, 40, 40, 48), 17  # 2.36e9 bytes a block, two blocks
    assert tl.tm_spinor_bytes_il(L, 16) > 2 ** 31 - 1
    U = torch.from_numpy(synth.gauge_field(L, 3, device="cuda").view(np.float64)).cuda()
    op = tl.Operator(L, 0.16, 0.01, U, recon=0)
    del U
    eta, x = tl.empty_field_il(L, n), tl.empty_field_il(L, n)
    x.fill_(0x7b)  # what was there must not matter
    tl.z4_noise_il(L, eta, tl.F16, 9, 0, n)
    for true_residual in (False, True):  # with b kept apart from r or not
        _, stats = tl.tm_cg_solve_il(op, x, eta, n, tl.cg_params(1e-2, 200, tl.CG_PLAIN, prec=tl.F16, schur=True,
                                                                 true_residual=true_residual))
        assert all(q["status"] == 0 and q["rel_res"] <= 1e-2 for q in stats)
    # the recursion's residual and the one recomputed in FP16 agree to the rounding of the vectors
    assert all(q["true_res"] <= 2e-2 for q in stats)
    op.close()
