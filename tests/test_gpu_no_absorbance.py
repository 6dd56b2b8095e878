"""Pixels whose global moments hold no absorbance although their samples do
(moments of other pieces, a cleared slab): nothing lies in front, so T = 1 and
every sample counts with its opacity, for every moment set and volume kind,
in the passes that take two points at once as in the one-point form of the
per-piece images."""
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


SCENES = {
    "grid": lambda: scenes.blobs512(width=150, height=61, n_pieces=1, n=48),      # windows
    "grid_odd": lambda: scenes.blobs512(width=21, height=19, n_pieces=1, n=33),   # direct loads
    "octree": lambda: scenes.amr_blobs(base=3, max_level=2, width=37, height=41, n_pieces=1),
    "mesh": lambda: scenes.tet_mesh(n=7, n_pieces=1, width=31, height=22),
}
SETS = [("power4", "f32", 5e-5), ("power6", "f32", 5e-5), ("power8", "f32", 5e-5), ("trig6", "f16", 2e-3),
        ("trig8", "bf16", 2e-2)]


def _blend(pkg, vol, sc, glob, mode):
    col = pkg.Volume.color_buffer(sc.views).fill_(7.0)
    vol.reconstruct_blend(sc.views, glob, col, mode=mode)
    n = vol.stats()["samples_pass2"]
    vol.synchronize()
    return col, n


@pytest.mark.parametrize("name", list(SCENES))
def test_no_absorbance_blends_every_sample(pkg, name):
    """A cleared slab says T = 1 in every moment set: the same colours, those of the one-point form."""
    import torch
    first = None
    for ms, storage, bias in SETS:
        sc = SCENES[name]()
        sc.moment_set, sc.storage, sc.moment_bias = ms, storage, bias
        vol = pkg.Volume(sc)
        glob = vol.moments_for(sc.views)
        one, n1 = _blend(pkg, vol, sc, glob, pkg.MBOIT_COLOR_PER_PIECE)
        col, n2 = _blend(pkg, vol, sc, glob, pkg.MBOIT_COLOR_REDUCED)
        assert n1 == n2 > 0 and (col.view(-1, 4)[:, 3] > 0).any()
        assert torch.equal(col.view(torch.int32), one.view(torch.int32)), ms
        first = col if first is None else first
        assert torch.equal(col.view(torch.int32), first.view(torch.int32)), ms
        vol.close()


@pytest.mark.parametrize("ms, storage, bias", SETS)
@pytest.mark.parametrize("name", list(SCENES))
def test_cleared_pixels_among_others(pkg, name, ms, storage, bias):
    """Every third pixel's absorbance cleared: lanes with and without a frame in one warp."""
    import torch
    sc = SCENES[name]()
    sc.moment_set, sc.storage, sc.moment_bias = ms, storage, bias
    vol = pkg.Volume(sc)
    glob = vol.moments_for(sc.views)
    vol.render_moments(sc.views, glob)
    npx = sc.views[0].width * sc.views[0].height
    glob[:npx:3] = 0.0   # the plane of b0 comes first
    one, n1 = _blend(pkg, vol, sc, glob, pkg.MBOIT_COLOR_PER_PIECE)
    col, n2 = _blend(pkg, vol, sc, glob, pkg.MBOIT_COLOR_REDUCED)
    assert n1 == n2 > 0
    assert torch.equal(col.view(torch.int32), one.view(torch.int32))
    assert np.isfinite(col.cpu().numpy()).all()
    vol.close()
