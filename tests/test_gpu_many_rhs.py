"""More right-hand sides than one launch of the right-hand-side kernel takes
(32): the polarizations of each equal, bit for bit, those of a solve of its own."""
import numpy as np
import pytest

from paper_0704_0037_gb300 import dda as _dda  # noqa: F401  (the binding imports without a GPU)
from paper_0704_0037_gb300 import inputs

from gpu_util import need_gpu, twin
from test_gpu_batch import _orientations

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("half", [16, 17, 33])
def test_each_right_hand_side_as_alone(half):
    torch, dda = need_gpu()
    p, _ = twin(inputs.ellipsoid(7, 6, 5), [1.5 + 0.02j], 0.5)
    prop, pol = _orientations(half, 3)
    opts = dict(solver=dda.DDA_QMR_CS, pol=dda.DDA_CLDR, prec=dda.DDA_FP64, tol=1e-9, maxiter=200)
    with p:
        dda.dda_build_Dmatrix(p.h, dda.DDA_FP64)
        P = torch.zeros((2 * half, 3, p.n_occ), dtype=torch.complex128, device="cuda")
        st, info = dda.dda_solve_batch(p.h, opts, prop, pol, P)
        assert st == dda.DDA_OK, info
        for r in sorted({0, 1, 30, 31, min(32, 2 * half - 1), 2 * half - 1}):
            Q = torch.zeros((1, 3, p.n_occ), dtype=torch.complex128, device="cuda")
            st, one, _ = dda.dda_solve(p.h, opts, prop[r:r + 1], pol[r:r + 1], Q)
            assert st == dda.DDA_OK and one[0]["iters"] == info[r]["iters"]
            assert torch.equal(Q[0], P[r]), r


def test_right_hand_sides_fit_the_memory_of_one_phase_table():
    """Phase tables of all right-hand sides at once take more memory than one
    after the other: a solve that fits a memory limit with one table is taken,
    with the same polarizations."""
    torch, dda = need_gpu()
    occ = inputs.ellipsoid(40, 14, 13)
    prop = inputs.random_unit_vectors(3, 12)
    pol = np.array([inputs.perpendicular_pols(a)[0] for a in prop])
    opts = dict(solver=dda.DDA_QMR_CS, pol=dda.DDA_LDR, prec=dda.DDA_FP64, tol=1e-6, maxiter=100, inner_tol=1e-4)
    dda.dda_release_cached_memory()
    table = 16 * sum(occ.shape)
    out, used = [], 0
    try:
        # all it can use; short of that (the FFT buffers of fewer right-hand sides);
        # short of that by the tables of all but one
        for short in (None, 1, 11 * table):
            with dda.Particle(occ, [1.2], 0.4) as p:
                dda.dda_build_Dmatrix(p.h, dda.DDA_FP64)
                P = torch.zeros((12, 3, p.n_occ), dtype=torch.complex128, device="cuda")
                live = dda.dda_memory_in_use()[0]
                # (a limit releases the cache, whose blocks may be larger than asked)
                dda.dda_set_memory_limit(live + used - short if short else 1 << 40)
                st, info = dda.dda_solve_batch(p.h, opts, prop, pol, P)
                assert st == dda.DDA_OK, info
                used = dda.dda_memory_in_use()[0] - live
                out.append(P.cpu().numpy())
            dda.dda_set_memory_limit(0)
    finally:
        dda.dda_set_memory_limit(0)
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
