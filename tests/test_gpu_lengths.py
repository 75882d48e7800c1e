"""Complex64 register-resident passes of the 7-smooth padded lengths between
the compiled lengths of all precisions: every length on every axis (the other
axes short), at its largest and smallest number of cells, and two boxes with
three of them; products and adjoint products against the oracle, and bit for
bit over repeats.  Tolerance: complex64 line transforms round at about
6e-8 log2(M) of the vector's norm; 2e-6 is the suite's bound of the same
arithmetic on other lengths with a factor of 5 to spare."""
import numpy as np
import pytest

from oracle.fft_matvec import matvec_fft
from paper_0704_0037_gb300 import inputs

from gpu_util import need_gpu, rel_l2, twin

pytestmark = pytest.mark.gpu

LENGTHS = {135: (65, 68), 140: (69, 70), 144: (71, 72), 147: (73, 74), 150: (75, 75), 160: (76, 80),
           162: (81, 81), 168: (82, 84), 175: (85, 88), 180: (89, 90), 189: (91, 95), 280: (136, 140),
           288: (141, 144), 294: (145, 147), 300: (148, 150), 315: (151, 158), 320: (159, 160),
           324: (161, 162), 336: (163, 168), 350: (173, 175), 360: (176, 180), 375: (181, 188),
           378: (189, 189)}


def _check(occ, grid_axis=None, length=None):
    torch, dda = need_gpu()
    p, prob = twin(occ, [1.3 + 0.02j], 0.5)
    with p:
        if length is not None:
            assert p.grid[grid_axis] == length
        dda.dda_build_Dmatrix(p.h, dda.DDA_FP32_REFINED)
        dda.dda_set_beta(p.h, dda.DDA_CLDR, [(0.6, 0.0, 0.8)] * 2, [(0.8, 0.0, -0.6)] * 2)
        x = inputs.random_vectors(13, 2, p.n_occ)
        xd = torch.from_numpy(x).to("cuda", torch.complex64)
        out = []
        for f in (dda.dda_matvec, dda.dda_matvec_adjoint, dda.dda_matvec):
            yd = torch.empty_like(xd)
            f(p.h, dda.DDA_FP32_REFINED, xd, yd, 2)
            out.append(yd.cpu().numpy())
    assert np.array_equal(out[0], out[2])
    beta = prob.beta("cldr", (0.6, 0.0, 0.8), (0.8, 0.0, -0.6))
    for r in range(2):
        assert rel_l2(out[0][r], matvec_fft(prob.occ, beta, prob.dmat(), x[r])) <= 2e-6
        assert rel_l2(out[1][r], matvec_fft(prob.occ, beta, prob.dmat(), x[r], conj=True)) <= 2e-6


@pytest.mark.parametrize("length", sorted(LENGTHS))
def test_length_on_each_axis(length):
    for n in sorted(set(LENGTHS[length])):
        for axis, box in enumerate(((n, 5, 4), (3, n, 5), (4, 3, n))):
            _check(inputs.random_occupancy(*box, fill=0.6, seed=n), axis, length)


@pytest.mark.parametrize("box", [(66, 90, 71), (95, 74, 82)])
def test_three_lengths(box):
    _check(inputs.ellipsoid(*box))


@pytest.mark.parametrize("length", [n for n in sorted(LENGTHS) if n % 2])
def test_odd_z_length_with_16_byte_rows(length):
    """x padded to an even length: the z pass stages its tile, which follows a
    table of an odd number of elements, in 16-byte copies."""
    n = LENGTHS[length][1]
    _check(inputs.random_occupancy(16, 5, n, fill=0.6, seed=n), 2, length)
