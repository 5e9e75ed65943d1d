"""Slots filled from a dense level, from the level below and from packed bricks: every voxel of
every brick (apron included) against the oracle's pyramid, and the value ranges and macro-cell spans
taken in the same pass by rendering with and without empty-space skipping."""
import numpy as np
import pytest
import torch

import synth
from _helpers import store_levels

pytestmark = pytest.mark.gpu

SKIP = 2  # VOL_RENDER_SKIP_EMPTY


@pytest.fixture(scope="module")
def P():
    import paper_2509_26213_gb300 as pkg
    pkg.build()
    from paper_2509_26213_gb300 import volume
    return volume


def brick_of(level, B, b):
    """(B+1)^3 voxels of brick b of a dense level, clamped to its edge."""
    ix = [np.minimum(np.arange(b[a] * B, b[a] * B + B + 1), level.shape[2 - a] - 1) for a in range(3)]
    return level[np.ix_(ix[2], ix[1], ix[0])]


@pytest.mark.parametrize("layout", ["quad", "compact"])
@pytest.mark.parametrize("dtype", ["u8", "u16", "f16", "f32"])
@pytest.mark.parametrize("brick,D", [(4, (9, 6, 5)), (8, (17, 8, 3)), (16, (33, 50, 17)), (32, (65, 31, 33)),
                                     (64, (65, 129, 20)), (128, (130, 127, 3))])
def test_slots_match_oracle(P, orc, layout, dtype, brick, D):
    rng = np.random.default_rng(brick)
    v = rng.random(D[::-1]).astype(np.float32) * (rng.random(D[::-1]) < 0.3)
    raw = {"u8": (v * 255).astype(np.uint8), "u16": (v * 65535).astype(np.uint16),
           "f16": v.astype(np.float16).view(np.uint16), "f32": v.astype(np.float32)}[dtype]
    levels = 3
    ref = store_levels(orc, raw, dtype, dtype, levels)
    vol = P.Volume(D, dtype, brick, levels, layout=layout)
    vol.upload_level(0, raw, dtype)
    vol.build_lod(0)
    bits = {"u8": np.uint8, "u16": np.uint16, "f16": np.uint16, "f32": np.uint32}[dtype]
    for l in range(levels):
        lev = np.ascontiguousarray(ref[l]).view(bits)
        nb = vol.level_bricks[l]
        for b in [(x, y, z) for z in range(nb[2]) for y in range(nb[1]) for x in range(nb[0])]:
            np.testing.assert_array_equal(vol.download_brick(l, b).view(bits), brick_of(lev, brick, b))
    # the same bricks sent one by one: the same slots, so the same image with and without skipping
    one = P.Volume(D, dtype, brick, levels, layout=layout)
    for l in range(levels):
        lev = np.ascontiguousarray(ref[l])
        nb = one.level_bricks[l]
        for b in [(x, y, z) for z in range(nb[2]) for y in range(nb[1]) for x in range(nb[0])]:
            one.upload_brick(l, b, np.ascontiguousarray(brick_of(lev, brick, b)), dtype)
            np.testing.assert_array_equal(one.download_brick(l, b).view(bits), brick_of(lev.view(bits), brick, b))
    tf = torch.from_numpy(synth.tf_ramp(alpha_start=0.5, alpha_max=0.3)).cuda()
    cams = [synth.seeded_orbit(D, 32, 24, 3), synth.seeded_orbit(D, 24, 32, 4)]
    for composite in ("dvr", "mop", "mip"):
        img = [w.render(cams, tf, {"lod_mode": 1, "composite": composite, "flags": f}).cpu().numpy()
               for w in (vol, one) for f in (0, SKIP)]
        for other in img[1:]:
            np.testing.assert_array_equal(other, img[0])


@pytest.mark.parametrize("dtype", ["f16", "f32"])
@pytest.mark.parametrize("layout", ["quad", "compact"])
def test_cells_with_infinities_and_nan(P, dtype, layout):
    """A cell with a NaN spans every entry, infinities are clamped: skipping changes no pixel."""
    D = (40, 33, 36)
    v = np.zeros(D[::-1], np.float32)
    v[8, 8, 8], v[20, 16, 24], v[30, 5, 39], v[35, 32, 0] = np.nan, np.inf, -np.inf, 1.0
    raw = v if dtype == "f32" else v.astype(np.float16).view(np.uint16)
    vol = P.Volume(D, dtype, 32, 2, layout=layout)
    vol.upload_level(0, raw, dtype)
    vol.build_lod(0)
    tf = torch.from_numpy(synth.tf_ramp(alpha_start=0.5, alpha_max=0.3)).cuda()
    cams = [synth.seeded_orbit(D, 48, 40, 3)]
    for composite in ("dvr", "mop", "mip"):
        a, b = (vol.render(cams, tf, {"composite": composite, "flags": f}).cpu().numpy() for f in (0, SKIP))
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("shift", range(0, 16, 5))
@pytest.mark.parametrize("dtype,brick", [("u8", 64), ("u8", 4), ("u16", 16), ("f32", 8)])
def test_packed_bricks_at_any_byte(P, shift, dtype, brick):
    """Packed device bricks that begin at any element: the copy realigns them."""
    npdt = {"u8": np.uint8, "u16": np.uint16, "f32": np.float32}[dtype]
    n = (brick + 1) ** 3
    rng = np.random.default_rng(shift)
    src = rng.integers(0, 200, n + 16).astype(npdt)
    D = (brick, brick, brick)
    vol = P.Volume(D, dtype, brick, 1, layout="compact")
    dev = torch.from_numpy(src.view(np.uint8)).cuda()
    off = shift * np.dtype(npdt).itemsize
    import ctypes
    from paper_2509_26213_gb300 import _capi as C
    b = (ctypes.c_int32 * 3)(0, 0, 0)
    C.check(vol.lib.vol_upload_brick(vol.h, 0, b, ctypes.c_void_p(dev.data_ptr() + off), C.DTYPES[dtype], 1), vol.h)
    np.testing.assert_array_equal(vol.download_brick(0, (0, 0, 0)).reshape(-1), src[shift:shift + n])
