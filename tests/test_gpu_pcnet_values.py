"""Values at the ends of the number types in the learned preconditioner's apply
pass: z = v + rms(v) N(v / rms(v)).

With zero biases and no weight on the occupancy channel the network is
homogeneous of degree 1 in the six field channels, so its output for tiny
features follows from that for features of 1."""
import numpy as np
import pytest

from paper_0704_0037_gb300 import inputs

from gpu_util import need_gpu, rel_l2
from test_gpu_pcnet import LAYERS

pytestmark = pytest.mark.gpu


def _pack(layers):
    return np.concatenate([np.concatenate([W.ravel(), b.ravel()]) for W, b in layers]).astype(np.float32)


def _zeros():
    return [(np.zeros((co, ci, k, k, k), np.float32), np.zeros(co, np.float32)) for ci, co, k in LAYERS]


def _field_weights(scale=1.0):
    """He-normal weights, zero biases, none on the occupancy; layer 0 times scale."""
    rng = np.random.default_rng(4)
    out = [(rng.standard_normal(W.shape) * np.sqrt(2.0 / W[0].size), b) for W, b in _zeros()]
    out[0][0][:, 6] = 0.0
    return _pack([(W * (scale if i == 0 else 1.0), b) for i, (W, b) in enumerate(out)])


def _apply(dda, torch, occ, w, v):
    with dda.Particle(occ, [1.5], 0.4) as p:
        net = dda.PcNet(0)
        net.set_weights(w)
        z = torch.empty((3, p.n_occ), dtype=torch.complex128, device="cuda")
        net.apply(p.h, torch.from_numpy(np.ascontiguousarray(v)).cuda(), z)
        out = z.cpu().numpy()
        net.close()
    return out


def test_field_whose_square_underflows_gives_zero_features():
    """|v|^2 sums to zero for v of 1e-170: rms(v) = 0, zero features, N(v) = v, and
    finite gradients of a training step."""
    torch, dda = need_gpu()
    occ = inputs.cube(10, 9, 8)
    v = inputs.random_vectors(3, 1, occ.size)[0] * 1e-170
    assert np.array_equal(_apply(dda, torch, occ, _field_weights(), v), v)
    with dda.Particle(occ, [1.5], 0.4) as p:
        net = dda.PcNet(0)
        r = torch.from_numpy(v).cuda()
        z, e = torch.empty_like(r), torch.from_numpy(inputs.random_vectors(4, 1, occ.size)[0]).cuda()
        assert abs(net.train_step(p.h, r, e, z, 1e-4) - 1.0) <= 1e-12
        assert np.array_equal(z.cpu().numpy(), v) and np.isfinite(net.grads()).all()
        net.close()


def test_cell_sums_keep_the_bits_of_their_fields():
    """Cells whose children cancel to 2^-52 of their size: the sum is exact in the
    fields' 53 bits and lost in 48.  The layer behind it makes 1 of it again."""
    torch, dda = need_gpu()
    n = 12
    occ = inputs.cube(n, n, n)
    ijk = np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1)[..., ::-1].reshape(-1, 3)   # x fastest
    first, second = (ijk % 2 == [0, 0, 0]).all(1), (ijk % 2 == [1, 0, 0]).all(1)
    v = np.zeros((3, n ** 3), complex)
    v[0, first], v[0, second] = 1 + (2 ** 28 + 1) * 2.0 ** -52, -(1 + 2 ** 28 * 2.0 ** -52)
    one = np.zeros((3, n ** 3), complex)
    one[0] = 1.0                                               # every feature 1 / rms
    rms, rms1 = (np.sqrt((np.abs(a) ** 2).mean()) for a in (v, one))
    got = (_apply(dda, torch, occ, _field_weights(2.0 ** 52), v) - v) / rms * (8 * rms)
    ref = (_apply(dda, torch, occ, _field_weights(), one) - one) / rms1 * rms1
    assert rel_l2(got, ref) <= 1e-5


@pytest.mark.parametrize("value", [1e-40, -3e-45, 2e-38, 0.0, 1.5, np.float32(3.4e38)])
def test_output_of_any_size_reaches_z(value):
    """The last layer's bias alone: z = v + rms value, subnormal floats included."""
    torch, dda = need_gpu()
    occ = inputs.cube(5, 4, 6)
    v = np.zeros((3, occ.size), complex)
    v[1, 7] = 2.0
    w = _zeros()
    w[6][1][:] = value
    z = _apply(dda, torch, occ, _pack(w), v)
    rms = np.sqrt((np.abs(v) ** 2).mean())
    b = float(np.float32(value))
    assert (np.abs(z - (v + rms * b * (1 + 1j))) <= 1e-14 * (np.abs(v) + rms * abs(b))).all()


def test_infinite_activation_stays_non_finite():
    """An overflow in the first layer, all weights positive: the output is infinite
    (a NaN on the way would come out of the next relu as 0)."""
    torch, dda = need_gpu()
    occ = inputs.cube(9, 8, 10)
    w = [(np.full_like(W, 0.01), b) for W, b in _zeros()]
    w[0][1][3] = np.inf
    v = inputs.random_vectors(3, 1, occ.size)[0]
    assert not np.isfinite(_apply(dda, torch, occ, _pack(w), v)).any()


@pytest.mark.parametrize("value", [3.4e38, 3.3895e38, 3.3e38, 1.2345678e20, 7.7e-30])
def test_activation_up_to_the_largest_float_is_kept(value):
    """One channel of the first layer through the skip connection, a power of two
    and a one: values that bf16 would round to infinity keep their 24 bits."""
    torch, dda = need_gpu()
    occ = inputs.cube(7, 6, 5)
    w = _zeros()
    w[0][1][0] = value
    scale = 2.0 ** -min(120, round(np.log2(value)))
    w[5][0][0, 32, 1, 1, 1] = scale
    w[6][0][:, 0] = 1.0
    v = inputs.random_vectors(3, 1, occ.size)[0]
    rms = np.sqrt((np.abs(v) ** 2).mean())
    got = (_apply(dda, torch, occ, _pack(w), v) - v) / rms
    ref = float(np.float32(value)) * scale * (1 + 1j)
    assert np.abs(got - ref).max() <= 1e-6 * abs(ref)
