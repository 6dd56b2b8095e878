"""Octree marches by brick words (aligned octrees without holes) against the
general march: a hole that no ray meets sends the same octree to the general
kernels, which must give the same bits; an octree whose coarse leaf is not
aligned to its size takes the general march and is held to the oracle."""
import numpy as np
import pytest

import oracle
import scenes
from tests.test_gpu_parity import assert_moments_close, assert_rgba_close, unpack_color, unpack_moments

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    import __graft_entry__
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    import paper_2501_12581_gb300 as p
    return p


def _view(D, width, height):
    """An orthographic window along z over the middle of the domain and past its x faces' inner half: no ray
    comes near the corner columns."""
    return scenes.View(np.array([D / 2, D / 2, -D], np.float32), np.array([1, 0, 0], np.float32),
                       np.array([0, 1, 0], np.float32), np.array([0.05, 0.03, 1.0], np.float32), width, height,
                       scenes.ORTHO, np.float32(0.6 * D), np.float32(0.6 * D), np.float32(0.5 * D), np.float32(3 * D))


@pytest.mark.parametrize("ms, storage, bias", [("power4", "f32", 5e-5), ("power8", "f32", 1e-3), ("trig6", "f16", 2e-3)])
@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("level, size", [(2, (45, 37)), (1, (33, 64)), (0, (8, 4))])
def test_bricks_equal_general_march(pkg, level, size, adaptive, ms, storage, bias):
    import torch
    out = []
    for hole in (False, True):
        sc = scenes.amr_blobs(base=5, max_level=level, width=8, height=8, n_pieces=3)
        sc.adaptive_step, sc.moment_set, sc.storage, sc.moment_bias = adaptive, ms, storage, bias
        if hole:
            keep = ~(sc.leaves[:, :3] == 0).all(1)
            assert keep.sum() == len(keep) - 1
            sc.leaves, sc.values, sc.piece_of_leaf = sc.leaves[keep], sc.values[keep], sc.piece_of_leaf[keep]
        sc.views = [_view(sc.finest_cells, *size), scenes.perspective_view(sc.dims, (0.1, -0.2, 1.0), 21, 13, fov_deg=7.0)]
        vol = pkg.Volume(sc)
        mom, col = vol.moments_for(sc.views), pkg.Volume.color_buffer(sc.views)
        res = []
        for launches in ((1, 2) if ms == "power4" else (2,)):
            vol.set_frame_launches(launches)
            vol.render_frame(sc.views, mom, col)
            res += [mom.clone(), col.clone()]
        vol.render_moments(sc.views, mom)
        vol.reconstruct_blend(sc.views, mom, col)
        vol.synchronize()
        st = vol.stats()
        out.append((res + [mom.clone(), col.clone()], st["samples_pass1"], st["samples_pass2"]))
        vol.close()
    assert out[0][1:] == out[1][1:] and out[0][1] > 0
    for a, b in zip(out[0][0], out[1][0]):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))


def test_unaligned_octree_against_oracle(pkg):
    import torch
    D, j = 32, np.arange(9.0)
    f = lambda x, y, z: 0.3 + x / 64 + y / 48 + z / 80 + 0.2 * np.sin(x / 5) * np.cos(y / 7)  # noqa: E731
    leaves = [(8, 8, 8, 0)] + [(x, y, z, 1) for z in range(0, D, 8) for y in range(0, D, 8) for x in range(0, D, 8)
                               if not (8 <= x < 24 and 8 <= y < 24 and 8 <= z < 24)]
    leaves = np.array(leaves, np.int32)
    vals = np.empty((len(leaves), 9, 9, 9), np.float32)
    for i, (x, y, z, L) in enumerate(leaves):
        h = 2.0 if L == 0 else 1.0
        Z, Y, X = np.meshgrid(z + j * h, y + j * h, x + j * h, indexing="ij")
        vals[i] = f(X, Y, Z)
    sc = scenes.amr_blobs(base=4, max_level=0, width=40, height=33, n_pieces=3)
    sc.leaves, sc.values, sc.max_level, sc.finest_cells = leaves, vals, 1, D
    sc.piece_of_leaf = (np.arange(len(leaves)) % 3).astype(np.int32)
    sc.tf_range = (np.float32(vals.min()), np.float32(vals.max()))
    sc.views = [scenes.perspective_view(sc.dims, (0.57, 0.49, 0.66), 40, 33)]
    vol = pkg.Volume(sc)
    mom, col = vol.moments_for(sc.views), pkg.Volume.color_buffer(sc.views)
    vol.render_frame(sc.views, mom, col)
    vol.synchronize()
    torch.cuda.synchronize()
    ref = oracle.render_amr(sc, want=("moments", "mboit", "nsamples"))
    assert vol.stats()["samples_pass1"] == int(ref["nsamples"].sum())
    assert_moments_close(unpack_moments(mom, sc.views)[0][0], ref["moments"])
    assert_rgba_close(unpack_color(col, sc.views)[0][0], ref["mboit"])
    vol.close()
