"""dda_scatter under a cap on device memory: with room for the digit products'
workspace, for that of 512 directions at a time, and for the direct sums alone
the amplitudes agree to the sums' FP64 accuracy (1e-13 of the largest); with
less the call is refused and the handle stays usable."""
import numpy as np
import pytest

from paper_0704_0037_gb300 import inputs

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box,n_dir", [((40, 40, 40), 700), ((6, 70, 70), 520), ((30, 40, 20), 90)])
def test_scatter_fits_the_memory_it_is_given(box, n_dir):
    torch, dda = need_gpu()
    nx, ny, nz = box
    prop, pol = [[0.0, 0.0, 1.0]], [[1.0, 0.0, 0.0]]
    dirs = inputs.random_unit_vectors(3, n_dir)
    dda.dda_release_cached_memory()
    # tables of all directions, partial sums of the groups of rows
    rows, dblocks = ny * nz, (n_dir + 3) // 4
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    chunks = max(1, min((4 * sms + dblocks - 1) // dblocks, (rows + 31) // 32))
    chunks = -(-rows // -(-rows // chunks))
    direct = 16 * (n_dir + 1) * (nx + ny + nz) + 48 * chunks * n_dir + 72 * n_dir + 24
    try:
        with dda.Particle(inputs.cube(nx, ny, nz), [1.4 + 0.05j], 0.2) as p:
            P = torch.from_numpy(inputs.random_vectors(3, 1, p.n_occ)).cuda()
            live = {}
            F = {}
            for name, room in (("none", None), ("least", direct), ("blocks", 7 << 20), ("short", direct // 2)):
                with dda.Particle(inputs.cube(nx, ny, nz), [1.4 + 0.05j], 0.2) as q:
                    _, q0 = dda.dda_scatter(q.h, dda.DDA_LDR, P, prop, pol, dirs[:0])   # beta, Q sums
                    live0 = dda.dda_memory_in_use()[0]
                    if room is not None:
                        dda.dda_set_memory_limit(live0 + room)
                    try:
                        if name == "short":
                            with pytest.raises(dda.DDAError) as ei:
                                dda.dda_scatter(q.h, dda.DDA_LDR, P, prop, pol, dirs)
                            assert ei.value.status == dda.DDA_ERR_OOM
                            dda.dda_set_memory_limit(0)
                        F[name], qs = dda.dda_scatter(q.h, dda.DDA_LDR, P, prop, pol, dirs)
                        assert np.array_equal(qs[:, :2], q0[:, :2])
                        live[name] = dda.dda_memory_in_use()[0] - live0
                    finally:
                        dda.dda_set_memory_limit(0)
            assert live["least"] <= direct < live["none"] == live["short"]
            for name in ("least", "blocks"):
                assert np.abs(F[name] - F["none"]).max() <= 1e-13 * np.abs(F["none"]).max()
            assert np.array_equal(F["short"], F["none"])
    finally:
        dda.dda_set_memory_limit(0)
