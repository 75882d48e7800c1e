"""The last operation of a product, y = x - beta u: with a refractive index close
to 1 the interaction is 1e-3 of x and less, so that a complex64 y carries the
one rounding of the difference and nothing else that shows.  Against the FP64
product of the same x its error is that of rounding the exact result to
complex64; a second rounding at the size of x (beta has both parts) would make
it 1.41 times as large.  Lattices of the fused planes, of the passes per axis
(by rows and not) and of the Stockham passes, forward and adjoint."""
import numpy as np
import pytest

from paper_0704_0037_gb300 import inputs

from gpu_util import need_gpu, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box", [(16, 16, 30), (24, 40, 40), (36, 60, 13), (50, 20, 20), (70, 15, 14), (130, 14, 13),
                                 (150, 13, 13), (6, 30, 30)])
def test_complex64_product_rounds_the_difference_once(box):
    torch, dda = need_gpu()
    occ = inputs.random_occupancy(*box, fill=0.6, seed=box[0])
    with dda.Particle(occ, [1.001 + 0.0008j], 0.45) as p:
        dda.dda_build_Dmatrix(p.h, dda.DDA_FP32_REFINED)
        dda.dda_set_beta(p.h, dda.DDA_CM, [(0.0, 0.0, 1.0)], [(1.0, 0.0, 0.0)])
        x = torch.from_numpy(inputs.random_vectors(5, 1, p.n_occ)).to("cuda", torch.complex64)
        for f in (dda.dda_matvec, dda.dda_matvec_adjoint):
            y, y64 = torch.empty_like(x), torch.empty_like(x, dtype=torch.complex128)
            f(p.h, dda.DDA_FP32_REFINED, x, y, 1)
            f(p.h, dda.DDA_FP64, x.to(torch.complex128), y64, 1)
            ref = y64.cpu().numpy()
            assert 1e-5 <= rel_l2(x.cpu().numpy(), ref) <= 1e-2
            assert rel_l2(y.cpu().numpy(), ref) <= 1.1 * rel_l2(ref.astype(np.complex64), ref)
