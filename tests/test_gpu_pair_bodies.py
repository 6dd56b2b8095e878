"""Pass 2 two points at a time against the one-point bodies: a volume of one
piece, whose per-piece image takes every sample through the one-point form, and
its frames (from the sample cache) and reduced split calls (which march again),
in windows of a grid and by direct loads, in an octree by brick words and by
leaves, and in a mesh.  Raw sums, the same bits, for every moment set and for
transfer functions on both sides of an absorbance of 1/4 a step (where the
opacity changes form) and across it."""
import numpy as np
import pytest

import scenes

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


def _octree(hole):
    sc = scenes.amr_blobs(base=3, max_level=2, width=43, height=41, n_pieces=1)
    if hole:   # general march
        sc.leaves, sc.values, sc.piece_of_leaf = sc.leaves[1:], sc.values[1:], sc.piece_of_leaf[1:]
    return sc


SCENES = {
    "grid_dense": lambda: scenes.blobs512(width=150, height=61, n_pieces=1, n=48),    # 16-byte windows
    "grid_dense_odd": lambda: scenes.blobs512(width=143, height=50, n_pieces=1, n=45),
    "grid_sparse": lambda: scenes.blobs512(width=21, height=19, n_pieces=1, n=64),    # direct loads
    "octree": lambda: _octree(False),
    "octree_hole": lambda: _octree(True),
    "mesh": lambda: scenes.tet_mesh(n=7, n_pieces=1, width=31, height=22),
}


def _opacities(sc, kind):
    """Largest absorbance of one step below 1/4, at least 1/4 everywhere, or both sides."""
    sc.tf = sc.tf.copy()
    quarter = -np.expm1(-0.25 / sc.step)       # the opacity whose step absorbs 1/4
    ramp = np.linspace(0.0, 1.0, 256)
    lo, hi = {"thin": (0.0, 0.9 * quarter), "thick": (1.05 * quarter, 0.95), "both": (0.0, 0.95)}[kind]
    sc.tf[:, 3] = (lo + (hi - lo) * ramp ** 2).astype(np.float32)


@pytest.mark.parametrize("ms, storage, bias", [("power4", "f32", 5e-5), ("power6", "f32", 5e-5), ("power8", "f32", 5e-5),
                                               ("trig6", "f16", 2e-3), ("trig8", "bf16", 2e-2)])
@pytest.mark.parametrize("opacity", ["thin", "thick", "both"])
@pytest.mark.parametrize("name", list(SCENES))
def test_pairs_equal_one_point_bodies(pkg, name, opacity, ms, storage, bias):
    import torch
    sc = SCENES[name]()
    sc.moment_set, sc.storage, sc.moment_bias = ms, storage, bias
    _opacities(sc, opacity)
    vol = pkg.Volume(sc, flags=pkg.MBOIT_FLAG_RAW_SUM)
    glob, one = vol.moments_for(sc.views), pkg.Volume.color_buffer(sc.views)
    vol.render_moments(sc.views, glob)
    vol.reconstruct_blend(sc.views, glob, one, mode=pkg.MBOIT_COLOR_PER_PIECE)
    n = vol.stats()["samples_pass2"]
    vol.synchronize()
    assert n > 0 and np.isfinite(one.cpu().numpy()).all()
    col = pkg.Volume.color_buffer(sc.views)
    for mode in (pkg.MBOIT_COLOR_REDUCED, pkg.MBOIT_COLOR_RESOLVED):
        vol.reconstruct_blend(sc.views, glob, col.fill_(7.0), mode=mode)
        assert vol.stats()["samples_pass2"] == n
        vol.synchronize()
        assert torch.equal(col.view(torch.int32), one.view(torch.int32))
    for launches in (1, 2) if ms == "power4" else (2,):
        vol.set_frame_launches(launches)
        mom = vol.moments_for(sc.views)
        vol.render_frame(sc.views, mom, col.fill_(7.0))
        assert vol.stats()["samples_pass2"] == n
        vol.synchronize()
        assert torch.equal(mom.view(torch.int32), glob.view(torch.int32))
        assert torch.equal(col.view(torch.int32), one.view(torch.int32))
    vol.close()
