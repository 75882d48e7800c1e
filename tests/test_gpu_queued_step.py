"""A solver's step is queued before the scalars of the one before it are read;
when the solve has ended, nothing of the queued step may run: the z passes of a
traced solve take the time of the products it reports."""
import numpy as np
import pytest

from paper_0704_0037_gb300 import inputs

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solver", ["qmr_cs", "bicg_cs", "bicgstab", "cgnr"])
def test_no_product_after_the_end_of_a_solve(solver):
    torch, dda = need_gpu()
    occ = inputs.cube(61, 45, 52)
    prop, pol = [[0.0, 0.0, 1.0]], [[1.0, 0.0, 0.0]]
    with dda.Particle(occ, [1.1], 0.3) as p:
        dda.dda_build_Dmatrix(p.h, dda.DDA_FP64)
        dda.dda_set_beta(p.h, dda.DDA_LDR, prop, pol)
        P = torch.zeros((1, 3, p.n_occ), dtype=torch.complex128, device="cuda")
        y = torch.empty_like(P)
        x = torch.from_numpy(inputs.random_vectors(3, 1, p.n_occ)).cuda()

        def z_ms(f):
            dda.dda_trace(p.h, 1)
            out = f()
            torch.cuda.synchronize()
            t = dda.dda_trace_read(p.h)
            dda.dda_trace(p.h, 0)
            return sum(ms for k, (ms, _) in t.items() if k.startswith("p3_")), out

        for _ in range(3):
            dda.dda_matvec(p.h, dda.DDA_FP64, x, y)
        one = z_ms(lambda: [dda.dda_matvec(p.h, dda.DDA_FP64, x, y) for _ in range(10)])[0] / 10
        for tol in (0.3, 0.1, 0.03, 1e-2, 1e-3):
            ms, (st, info, _) = z_ms(lambda: dda.dda_solve(p.h, dict(
                solver=dda.SOLVER[solver], pol=dda.DDA_LDR, prec=dda.DDA_FP64, tol=tol, maxiter=50), prop, pol, P))
            assert st == dda.DDA_OK
            assert ms <= (info[0]["matvecs"] + 0.5) * one, (tol, ms, one, info[0])
