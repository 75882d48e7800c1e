"""Complex64 products on small grids, whose x and y passes run fused per z plane:
every pair of plane lengths, planes and rows without dipoles, one and many
right-hand sides (whole planes and groups of columns), the z lengths that hold
the product in registers and one that does not, forward and adjoint, against
the oracle and bit for bit over right-hand sides.  Tolerance: complex64 line
transforms round at about 6e-8 log2(M) of the vector's norm, three axes and the
product; 2e-6 is the suite's bound of the same arithmetic on other lengths."""
import numpy as np
import pytest

from oracle.fft_matvec import matvec_fft
from paper_0704_0037_gb300 import inputs

from gpu_util import need_gpu, rel_l2, twin

pytestmark = pytest.mark.gpu

CELLS = {32: 16, 40: 20, 48: 23, 64: 32, 80: 39, 96: 47}


def _check(occ, nrhs, grid=None):
    torch, dda = need_gpu()
    p, prob = twin(occ, [1.3 + 0.02j], 0.5)
    with p:
        if grid is not None:
            assert tuple(p.grid[:2]) == grid
        dda.dda_build_Dmatrix(p.h, dda.DDA_FP32_REFINED)
        dda.dda_set_beta(p.h, dda.DDA_CLDR, [(0.6, 0.0, 0.8)] * nrhs, [(0.8, 0.0, -0.6)] * nrhs)
        x = inputs.random_vectors(13, 2, p.n_occ)[np.arange(nrhs) % 2]
        xd = torch.from_numpy(x).to("cuda", torch.complex64)
        out = []
        for f in (dda.dda_matvec, dda.dda_matvec_adjoint):
            yd = torch.empty_like(xd)
            f(p.h, dda.DDA_FP32_REFINED, xd, yd, nrhs)
            out.append(yd.cpu().numpy())
    beta = prob.beta("cldr", (0.6, 0.0, 0.8), (0.8, 0.0, -0.6))
    for r in range(min(nrhs, 2)):
        assert rel_l2(out[0][r], matvec_fft(prob.occ, beta, prob.dmat(), x[r])) <= 2e-6
        assert rel_l2(out[1][r], matvec_fft(prob.occ, beta, prob.dmat(), x[r], conj=True)) <= 2e-6
    for r in range(2, nrhs):
        assert np.array_equal(out[0][r], out[0][r - 2]) and np.array_equal(out[1][r], out[1][r - 2])


@pytest.mark.parametrize("mx", sorted(CELLS))
@pytest.mark.parametrize("my", sorted(CELLS))
def test_every_pair_of_plane_lengths(mx, my):
    _check(inputs.random_occupancy(CELLS[mx], CELLS[my], 7, fill=0.5, seed=mx + my), 1, (mx, my))


@pytest.mark.parametrize("nrhs", [1, 16])
@pytest.mark.parametrize("nz", [15, 19, 24, 31, 40, 48, 64, 70])
def test_z_lengths_and_groups_of_columns(nz, nrhs):
    _check(inputs.random_occupancy(37, 30, nz, fill=0.4, seed=nz), nrhs)


@pytest.mark.parametrize("nrhs", [1, 16])
def test_planes_and_rows_without_dipoles(nrhs):
    occ = inputs.random_occupancy(36, 31, 18, fill=0.3, seed=3)
    occ[4:9] = 0
    occ[:, 10:14] = 0
    occ[:, :, 20:25] = 0
    occ[0, :, :] = 0
    occ[0, 5, 7] = 1
    occ[-1, :, :] = 0
    occ[-1, -1, -1] = 1
    _check(occ, nrhs)


@pytest.mark.parametrize("mx", sorted(CELLS))
@pytest.mark.parametrize("my", sorted(CELLS))
def test_every_pair_of_plane_lengths_with_planes_to_fuse(mx, my):
    """25 planes: fused whatever the lengths (7, above, are for the shorter ones)."""
    _check(inputs.random_occupancy(CELLS[mx], CELLS[my], 25, fill=0.4, seed=mx + 2 * my), 1, (mx, my))


@pytest.mark.parametrize("box,nrhs,fused", [((47, 45, 21), 1, False), ((47, 45, 22), 1, True), ((47, 45, 10), 2, False),
                                            ((47, 45, 11), 2, True), ((30, 31, 10), 1, False),
                                            ((47, 23, 1), 1, True), ((16, 46, 2), 1, True)])
def test_line_between_fused_and_separate_passes(box, nrhs, fused):
    """The traced passes say which way a solve's products went; the products and
    their sums (x^T y) come from either."""
    torch, dda = need_gpu()
    occ = inputs.cube(*box)
    _check(occ, nrhs)
    with dda.Particle(occ, [1.3], 0.5) as p:
        dda.dda_build_Dmatrix(p.h, dda.DDA_FP32_REFINED)
        P = torch.zeros((nrhs, 3, p.n_occ), dtype=torch.complex128, device="cuda")
        dda.dda_trace(p.h, 1)
        st, info = dda.dda_solve_batch(p.h, dict(solver=dda.DDA_QMR_CS, pol=dda.DDA_LDR, prec=dda.DDA_FP32_REFINED,
                                                 tol=1e-6, maxiter=200, inner_tol=1e-4), [[0.0, 0.0, 1.0]] * nrhs,
                                       [[1.0, 0.0, 0.0]] * nrhs, P)
        names = set(dda.dda_trace_read(p.h))
        dda.dda_trace(p.h, 0)
        assert st == dda.DDA_OK and all(i["rel_res_true"] < 1e-6 for i in info)
        assert any(k.startswith("p2_") and k.endswith("c64") for k in names) != fused, names
