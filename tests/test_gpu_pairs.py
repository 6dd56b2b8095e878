"""Pass 2 two points at a time (frames, from the sample cache) against one point
at a time (the split calls march the volume again): the same bits, for every
moment set, at ray ends that fill no chunk, with pieces left out and where
some rays meet no absorbance."""
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


def _clear_half(sc):
    """A transfer function whose lower half is fully transparent."""
    sc.tf = sc.tf.copy()
    sc.tf[:150, 3] = 0.0
    return sc


SCENES = {
    "grid": lambda: scenes.blobs512(width=43, height=29, n_pieces=5, n=48),
    "grid_clear": lambda: _clear_half(scenes.blobs64(width=40, height=36)),
    "grid_tiny": lambda: scenes.blobs512(width=9, height=5, n_pieces=2, n=33),
    "octree": lambda: scenes.amr_blobs(base=3, max_level=2, width=37, height=41, n_pieces=4),
    "mesh": lambda: scenes.tet_mesh(n=7, n_pieces=3, width=31, height=22),
}


@pytest.mark.parametrize("ms, storage, bias", [("power4", "f32", 5e-5), ("power6", "f32", 5e-5), ("power8", "f32", 5e-5),
                                               ("trig6", "f16", 2e-3), ("trig8", "bf16", 2e-2)])
@pytest.mark.parametrize("name", list(SCENES))
def test_pairs_equal_single_points(pkg, name, ms, storage, bias):
    import torch
    sc = SCENES[name]()
    sc.moment_set, sc.storage, sc.moment_bias = ms, storage, bias
    vol = pkg.Volume(sc)
    frame, split = ((vol.moments_for(sc.views), pkg.Volume.color_buffer(sc.views)) for _ in range(2))
    vol.set_frame_launches(2)
    vol.render_frame(sc.views, *frame)
    nf = vol.stats()["samples_pass2"]
    vol.render_moments(sc.views, split[0])
    vol.reconstruct_blend(sc.views, *split)
    vol.synchronize()
    assert nf == vol.stats()["samples_pass2"] > 0
    assert np.isfinite(frame[1].cpu().numpy()).all()
    for a, b in zip(frame, split):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    vol.close()
