"""GPU parity of the far-field sums (exact digit products on the tensor cores)
with the oracle's direct sum, at the edges of their tiles: folded rows of one
cell, odd and even lengths, one and several inner chunks (72 folded cells
each), row blocks of 8 that are partly filled, lattices with more row blocks
than run at once, direction tiles of 32, and calls whose directions are taken in
several blocks of 8,192.

Tolerance: both sides evaluate the phases in FP64 (|phase| <= kd n: relative
error of a sum a few 1e-16 times kd n) and sum at FP64 accuracy: 1e-13 of the
largest amplitude leaves a factor of 20 at the largest case (kd n = 60)."""
import numpy as np
import pytest

from oracle import lattice, observables
from paper_0704_0037_gb300 import inputs

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

CASES = [  # nx, ny, nz, fill (0: full box), directions
    (1, 1, 1, 0, 1), (2, 1, 3, 0, 31), (5, 4, 4, 0, 32), (16, 3, 6, 0.4, 33), (15, 7, 5, 0.5, 64),
    (143, 3, 2, 0.7, 40), (144, 2, 3, 0, 5), (145, 3, 3, 0.3, 70), (300, 2, 2, 0.6, 45),
    (9, 33, 17, 0.2, 130),
    # more than 2 x 152 row blocks: a block's sums carried over several of them,
    # with one inner chunk and with two
    (6, 70, 70, 0, 34), (150, 50, 50, 0, 36),
]


@pytest.mark.parametrize("nx,ny,nz,fill,n_dir", CASES)
def test_farfield_matches_direct_sum(nx, ny, nz, fill, n_dir):
    torch, dda = need_gpu()
    occ = inputs.random_occupancy(nx, ny, nz, fill, seed=nx) if fill else inputs.cube(nx, ny, nz)
    occ[nz // 2, ny // 2, nx // 2] = 1
    pos = lattice.positions(occ > 0)
    prop, pol = [[0.0, 0.0, 1.0]] * 2, [[1.0, 0.0, 0.0], [0.0, 1.0, 0.0]]
    dirs = inputs.random_unit_vectors(n_dir, n_dir)
    if n_dir % 2:                       # the y-collapsed lattice of in-plane directions
        dirs[:, 1] = 0.0
    with dda.Particle(occ, [1.4 + 0.05j], 0.2) as p:
        x = inputs.random_vectors(3, 2, p.n_occ)
        x[1, 1] = 0.0                   # a component without any field
        x[1, 2] *= 10.0 ** np.linspace(-30, 0, p.n_occ)
        P = torch.from_numpy(x).cuda()
        F, _ = dda.dda_scatter(p.h, dda.DDA_LDR, P, prop, pol, dirs)
        again, _ = dda.dda_scatter(p.h, dda.DDA_LDR, P, prop, pol, dirs)
        assert np.array_equal(F, again)
        for r in range(2):
            ref = observables.farfield(x[r], pos, p.kd, dirs)
            assert np.abs(F[r] - ref).max() <= 1e-13 * np.abs(ref).max()


def test_farfield_nonfinite_input_stays_nonfinite():
    torch, dda = need_gpu()
    occ = inputs.cube(6, 5, 4)
    with dda.Particle(occ, [1.4], 0.2) as p:
        x = inputs.random_vectors(3, 1, p.n_occ)
        x[0, 0, 7] = np.nan
        x[0, 1, 9] = np.inf
        F, q = dda.dda_scatter(p.h, dda.DDA_LDR, torch.from_numpy(x).cuda(), [[0.0, 0.0, 1.0]],
                               [[1.0, 0.0, 0.0]], inputs.random_unit_vectors(1, 9))
        assert not np.isfinite(F).any() and not np.isfinite(q[0, 0])


def test_farfield_of_several_direction_blocks():
    """16,368 directions (8,192 + 8,176: a last block for which a plan of its own
    would not have fitted the first one's workspace) against the oracle at
    directions of both blocks, and against calls of one block."""
    torch, dda = need_gpu()
    nx, ny, nz, n_dir = 6, 70, 70, 16368
    occ = inputs.cube(nx, ny, nz)
    pos = lattice.positions(occ > 0)
    prop, pol = [[0.0, 0.0, 1.0]] * 2, [[1.0, 0.0, 0.0], [0.0, 1.0, 0.0]]
    dirs = inputs.random_unit_vectors(7, n_dir)
    with dda.Particle(occ, [1.4 + 0.05j], 0.2) as p:
        x = inputs.random_vectors(3, 2, p.n_occ)
        P = torch.from_numpy(x).cuda()
        F, q = dda.dda_scatter(p.h, dda.DDA_LDR, P, prop, pol, dirs)
        pick = [0, 31, 4095, 8191, 8192, 8193, 12000, n_dir - 1]
        for r in range(2):
            ref = observables.farfield(x[r], pos, p.kd, dirs[pick])
            assert np.abs(F[r][pick] - ref).max() <= 1e-13 * np.abs(ref).max()
        for d0, d1 in ((0, 8192), (8192, n_dir), (5000, 9000)):
            part, q1 = dda.dda_scatter(p.h, dda.DDA_LDR, P, prop, pol, dirs[d0:d1])
            assert np.abs(part - F[:, d0:d1]).max() <= 1e-13 * np.abs(F).max()
            assert np.array_equal(q[:, :2], q1[:, :2])      # Q sums: their table lies behind the plan


@pytest.mark.parametrize("nx", [31, 100, 144])
def test_farfield_row_is_as_exact_as_its_phases(nx):
    """One lattice row and directions whose phase arguments are exact in FP64: the
    error of a sum is that of its cosines and sines, each rounded to at most half
    a unit of 2^-53 (0.41 2^-53 rms per complex entry), in nx terms of random
    sign, and of the final roundings: below 0.55 2^-53 sqrt(nx) of the largest
    entry.  Digit products left out of the sum must not show."""
    torch, dda = need_gpu()
    kd, n_dir = 0.125, 96
    c = np.arange(1, n_dir + 1) / 128.0
    dirs = np.stack([c, np.zeros(n_dir), np.sqrt(1.0 - c * c)], axis=1)
    rng = np.random.default_rng(1)
    x = rng.uniform(-1, 1, (1, 3, nx)) + 1j * rng.uniform(-1, 1, (1, 3, nx))
    with dda.Particle(inputs.cube(nx, 1, 1), [1.4], kd) as p:
        F, _ = dda.dda_scatter(p.h, dda.DDA_LDR, torch.from_numpy(x).cuda(), [[0.0, 0.0, 1.0]],
                               [[1.0, 0.0, 0.0]], dirs)
    ph = np.outer(kd * c, np.arange(nx) - 0.5 * (nx - 1)).astype(np.longdouble)
    ref = -1j * np.longdouble(kd) ** 3 * ((np.cos(ph) - 1j * np.sin(ph)) @ x[0, 1].astype(np.clongdouble))
    err = np.abs(F.reshape(n_dir, 3)[:, 1] - ref).astype(float) / kd ** 3      # y: no projection
    assert np.sqrt((err ** 2).mean()) <= 0.55 * 2.0 ** -53 * np.sqrt(nx) * np.abs(x).max()
