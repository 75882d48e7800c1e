"""The learned preconditioner's kernels over lattice sizes: convolution tiles of
128 and 64 voxels by 40 to 8 channels, one to four groups of channels, one to
many blocks, partial tiles and cells on every axis, in the apply pass (tensor
cores) and in a training step (FP32 pipe), against the float64 restatement.

Tolerance of N(r) = z - r: every product is exact or correctly rounded, so the
error is that of seven layers' FP32 sums of up to 5,184 terms, 6e-8 sqrt(5184)
each when the roundings are independent: 7 * 4.3e-6 = 3e-5.  Gradients add the
relu masks that such an error flips (1e-3, as in test_gpu_pcnet)."""
import numpy as np
import pytest

from paper_0704_0037_gb300 import inputs

from gpu_util import need_gpu, rel_l2, twin
from test_gpu_pcnet import LAYERS, _reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box", [(4, 4, 4), (8, 3, 5), (17, 16, 33), (31, 34, 18), (70, 12, 9), (9, 66, 64),
                                 (64, 45, 37), (96, 64, 64)])
def test_forward_and_gradients_over_lattice_sizes(box):
    torch, dda = need_gpu()
    occ = inputs.random_occupancy(*box, fill=0.6, seed=box[0])
    p, prob = twin(occ, [1.6 + 0.02j], 0.45)
    net = dda.PcNet(seed=7)
    with p:
        r = inputs.random_vectors(31, 1, p.n_occ)[0]
        e = inputs.random_vectors(32, 1, p.n_occ)[0]
        rd, ed = torch.from_numpy(r).cuda(), torch.from_numpy(e).cuda()
        z_ref, params = _reference(torch, net.weights(), occ, r)
        n_ref = z_ref.detach().numpy() - r
        zd = torch.empty_like(rd)
        net.apply(p.h, rd, zd)
        assert rel_l2(zd.cpu().numpy() - r, n_ref) < 3e-5
        loss = net.train_step(p.h, rd, ed, zd, 1e-4)
        assert rel_l2(zd.cpu().numpy() - r, n_ref) < 3e-5
        et = torch.tensor(e)
        loss_ref = ((z_ref - et).abs() ** 2).sum() / (et.abs() ** 2).sum()
        assert abs(loss - loss_ref.item()) < 1e-5 * loss_ref.item()
        loss_ref.backward()
        g, o = net.grads(), 0
        for (W, b), (cin, cout, k) in zip(params, LAYERS):
            n = cout * cin * k ** 3
            assert rel_l2(g[o:o + n], W.grad.numpy().ravel()) < 1e-3, (cin, cout)
            assert rel_l2(g[o + n:o + n + cout], b.grad.numpy()) < 1e-3, (cin, cout)
            o += n + cout
    net.close()
