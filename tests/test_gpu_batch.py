"""The forward's batched decisions (a batch's samples decided by pairs, one brick lookup per batch,
one level per batch) at the sizes where a batch can go wrong: bricks smaller than a batch's reach
and steps longer than a brick, an axis too long for the 2^23 floor, level changes inside a batch,
rays that leave the volume inside a batch, a preview whose last brick is absent."""
import numpy as np
import pytest
import torch

import synth
from _helpers import AMB, TOL_FP32, compare, store_levels

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2509_26213_gb300 as pkg
    pkg.build()
    from paper_2509_26213_gb300 import volume
    return volume


def check(P, orc, D, dtype, brick, levels, layout, cams, params, seed=5):
    base = synth.blobs(D, seed, dtype="f32", nblobs=5, sigma=(3, 9), amp=(0.3, 1.0), noise=0.05, vmax=1.0)
    raw = {"u8": (base * 255).astype(np.uint8), "u16": (base * 65535).astype(np.uint16),
           "f16": base.astype(np.float16).view(np.uint16), "f32": base}[dtype]
    vol = P.Volume(D, dtype, brick, levels, layout=layout)
    vol.upload_level(0, raw, dtype)
    if levels > 1:
        vol.build_lod(0)
    tf = synth.tf_ramp(alpha_start=0.1, alpha_max=0.1)
    out, ns = vol.render(cams, torch.from_numpy(tf).cuda(), params, nsamples=True)
    out, ns = out.cpu().numpy(), ns.cpu().numpy()
    ovol = orc.Volume(store_levels(orc, raw, dtype, dtype, levels), dtype, brick)
    off = 0
    for cam in cams:
        n = cam["w"] * cam["h"]
        ref = orc.render(ovol, cam, tf, params, amb=AMB)
        err, bad, alt = compare(out[off:off + n], ref, TOL_FP32)
        assert len(bad) == 0, err
        off += n
    vol.close()


@pytest.mark.parametrize("dtype,layout", [("u8", "quad"), ("u16", "quad"), ("f16", "quad"), ("f32", "quad"),
                                          ("u8", "compact"), ("f16", "compact"), ("f32", "compact")])
@pytest.mark.parametrize("brick,step", [(4, 0.5), (4, 5.0), (8, 9.0), (32, 0.37), (64, 0.05), (128, 1.0)])
def test_batches_match_oracle(P, orc, dtype, layout, brick, step):
    D = (70, 37, 65)
    cams = [synth.seeded_orbit(D, 33, 21, 3), synth.look_at((30.0, 20.0, 31.0), (60.0, 30.0, 12.0), 24, 17, fov_deg=60.0)]
    check(P, orc, D, dtype, brick, 3, layout, cams, {"step": step, "et": 0.99, "lod_mode": 1})
    check(P, orc, D, dtype, brick, 1, layout, cams, {"step": step, "et": 0.99, "lod_mode": 0})


@pytest.mark.parametrize("bias", [-2, 0, 1, 3])
def test_level_changes_inside_a_batch(P, orc, bias):
    """A camera in the volume's corner with a wide field of view: every level within a few samples."""
    D = (96, 96, 96)
    cams = [synth.look_at((1.0, 2.0, 1.5), (80.0, 70.0, 90.0), 32, 24, fov_deg=100.0)]
    check(P, orc, D, "u16", 16, 6, "quad", cams, {"step": 2.0, "et": 0.99, "lod_mode": 1, "lod_bias": bias})


def test_axis_longer_than_the_floor_constant(P, orc):
    """An axis above 2^23 voxels takes the conversions instead of the floor by 2^23."""
    D = ((1 << 23) + 37, 3, 2)
    rng = np.random.default_rng(3)
    raw = rng.integers(0, 256, D[::-1], dtype=np.uint8)
    tf = synth.tf_ramp(alpha_start=0.1, alpha_max=0.3)
    params = {"step": 0.75, "et": 2.0, "lod_mode": 0}  # (below 2^24 samples on the diagonal)
    c = np.array([D[0] - 8.0, 1.5, 1.0])
    cam = synth.look_at(tuple(c + np.array([2.0, 9.0, 4.0])), tuple(c), 16, 12, fov_deg=60.0)
    vol = P.Volume(D, "u8", 4, 1)
    vol.upload_level(0, raw, "u8")
    out = vol.render(cam, torch.from_numpy(tf).cuda(), params).cpu().numpy()
    ref = orc.render(orc.Volume([raw], "u8", 4), cam, tf, params, amb=AMB)
    err, bad, _ = compare(out, ref, TOL_FP32)
    assert len(bad) == 0, err
    assert np.abs(out).max() > 0.01


def test_preview_ends_on_absent_bricks(P):
    """Nothing resident, no coarser level: every ray leaves the volume with nothing composited."""
    D = (40, 40, 40)
    vol = P.Volume(D, "u8", 16, 1, cache_bytes=1 << 20)
    tf = torch.from_numpy(synth.tf_ramp(alpha_start=0.1, alpha_max=0.1)).cuda()
    cam = synth.seeded_orbit(D, 24, 16, 2)
    bg = (0.25, 0.5, 0.75, 0.0)
    out, ns = vol.render(cam, tf, {"flags": 8, "bg": bg}, nsamples=True, check_incomplete=False)
    np.testing.assert_array_equal(out.cpu().numpy(), np.tile(np.float32(bg), (24 * 16, 1)))
    assert int(ns.max()) > 0
