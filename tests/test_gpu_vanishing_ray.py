"""A perspective view in which one pixel's direction vanishes (w + sx u + sy v =
0): that pixel has no ray and stays empty, and no call steps through the whole
lattice to find that out.

Time limit: the lattice has 2^22 points and a step of the search is a chain of
at least six dependent instructions of four cycles, so stepping through it
takes more than 2^22 * 24 cycles, 48 ms at 2.07 GHz; every call here takes well
under 2 ms, so 20 ms tell the two apart."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu
LIMIT_MS = 20.0


@pytest.fixture(scope="module")
def pkg():
    import torch
    import __graft_entry__
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    import paper_2501_12581_gb300 as p
    return p


W, H, PX, PY = 64, 33, 8, 16


def _view(D):
    """Looks along x from outside; sx = -47/64 and sy = 0 at pixel (PX, PY), exactly."""
    f = np.float32
    u = np.array([1, 0, 0], f)
    return scenes.View(np.array([-0.6 * D, 0.5 * D, 0.5 * D], f), u, np.array([0, 1, 0.3], f), f(47 / 64) * u, W, H,
                       scenes.PERSPECTIVE, f(1), f(1), f(0.01 * D), f(4 * D))


SCENES = {
    "grid": lambda: scenes.blobs512(width=8, height=8, n_pieces=4, n=64),
    "grid_odd": lambda: scenes.blobs512(width=8, height=8, n_pieces=4, n=45),
    "octree": lambda: scenes.amr_blobs(base=3, max_level=2, width=8, height=8, n_pieces=4),
    "mesh": lambda: scenes.tet_mesh(n=7, n_pieces=4, width=8, height=8),
}


@pytest.mark.parametrize("name", list(SCENES))
def test_vanishing_direction(pkg, name):
    import torch
    sc = SCENES[name]()
    D = float(sc.box[0]) if name == "mesh" else float(sc.dims[0] - 1)
    views = [_view(D)]
    vol = pkg.Volume(sc)
    K = sc.n_pieces
    mom, col = vol.moments_for(views), pkg.Volume.color_buffer(views)
    pm, pc = vol.moments_for(views, K), pkg.Volume.color_buffer(views, K)

    def frame(launches):
        vol.set_frame_launches(launches)
        vol.render_frame(views, mom, col)

    def split():
        vol.render_moments(views, mom)
        vol.reconstruct_blend(views, mom, col)

    def pieces(n):
        vol.render_moments(views, pm, pieces=list(range(n)), mode=pkg.MBOIT_MOMENTS_PER_PIECE)
        vol.reconstruct_blend(views, mom, pc, pieces=list(range(n)), mode=pkg.MBOIT_COLOR_PER_PIECE)

    calls = {"split": split, "frame 1": lambda: frame(1), "frame 2": lambda: frame(2), "own march": lambda: pieces(1),
             "one march": lambda: pieces(K), "sort-last": lambda: vol.render_sortlast(views, col)}
    if name != "mesh":
        calls["multi"] = lambda: pkg.Volume.render_frame_multi([vol], views, [0], mom, col)
    for what, call in calls.items():
        call()   # first call: graphs, cache
        vol.synchronize()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        call()
        b.record()
        vol.synchronize()
        torch.cuda.synchronize()
        assert a.elapsed_time(b) < LIMIT_MS, what
        img = (pc if "march" in what else col)[:W * H * 4].view(H, W, 4).cpu().numpy()
        assert np.isfinite(img).all() and (img[PY, PX] == 0).all() and (img[..., 3] > 0).sum() > 20, what
    vol.close()
