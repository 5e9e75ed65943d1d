"""dL/dvoxel through the gradient quads (many rays per voxel) against the direct reductions (few
rays): the same view's gradient, alone and beside copies of the view whose upstream gradient is
zero, which take the adjoint to the quads.  Each voxel sums the same terms in another order, so
the two differ by the rounding of binary32 sums: at most a few hundred terms per voxel, 2^-24
relative each, so 1e-4 of the largest gradient is far above it."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2509_26213_gb300 as pkg
    pkg.build()
    from paper_2509_26213_gb300 import volume
    return volume


@pytest.mark.parametrize("D,brick,levels", [((33, 18, 25), 16, 1), ((33, 18, 25), 8, 3), ((5, 4, 3), 4, 2), ((64, 64, 64), 32, 2)])
def test_quads_equal_direct(P, D, brick, levels):
    raw = synth.blobs(D, 3, dtype="f32", nblobs=5, sigma=(3, 6), amp=(0.3, 0.9), noise=0.05, vmax=1.0)
    vol = P.Volume(D, "f32", brick, levels)
    vol.upload_level(0, raw, "f32")
    if levels > 1:
        vol.build_lod(0)
    tf = torch.from_numpy(synth.tf_ramp(alpha_start=0.1, alpha_max=0.1)).cuda()
    w, h = 8, 6
    cam = synth.seeded_orbit(D, w, h, 3)
    params = {"step": 0.5, "lod_mode": int(levels > 1)}
    one = np.random.default_rng(1).standard_normal((w * h, 4)).astype(np.float32)
    got = []
    voxels = sum(np.prod(d) for d in vol.level_dims[:levels])
    many = int(np.ceil(8.0 * voxels / (w * h * max(D) / 0.5))) + 1
    for copies in (1, many):
        vol.render([cam] * copies, tf, params, grad=True)
        g = torch.zeros((copies * w * h, 4), device="cuda")
        g[:w * h] = torch.from_numpy(one).cuda()
        dvox = torch.full(raw.shape, 0.5, device="cuda")  # the adjoint adds to what is there
        dtf = torch.zeros((256, 4), device="cuda")
        vol.render_backward(g, dtf, dvox)
        got.append((dvox.cpu().numpy() - 0.5, dtf.cpu().numpy()))
    assert np.abs(got[0][0]).max() > 1e-3
    for a, b in zip(*got):
        np.testing.assert_allclose(a, b, rtol=0, atol=1e-4 * np.abs(a).max())
