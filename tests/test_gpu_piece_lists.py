"""Per-piece images of a short list of pieces: a piece whose box spans the
domain but which fills little of it keeps its own march, which skips the
other pieces' units, and does not pay for a walk of the whole volume.

Limit: the image of such a piece against the images of all pieces from one
march (which walks the whole volume and samples every point of it).  The walk
alone was measured at half of that (0.47 to 0.56), such a piece's own march at
a quarter; 0.4 tells them apart."""
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


def _grid(n):
    sc = scenes.blobs512(width=512, height=512, n_pieces=4, n=n)
    corners = np.zeros(sc.brick_dims[::-1], bool)
    corners[0, 0, 0] = corners[-1, -1, -1] = True
    return sc, corners.ravel()


def _octree():
    sc = scenes.amr_blobs(base=10, max_level=1, width=512, height=512, n_pieces=4)
    size = 8 << (sc.max_level - sc.leaves[:, 3:])
    return sc, (sc.leaves[:, :3] == 0).all(1) | (sc.leaves[:, :3] + size == sc.dims[0] - 1).all(1)


@pytest.mark.parametrize("name", ["grid", "grid_odd", "octree"])
def test_sparse_piece_keeps_its_own_march(pkg, name):
    import torch
    sc, corners = _octree() if name == "octree" else _grid(161 if name == "grid" else 160)
    pieces = "piece_of_leaf" if name == "octree" else "piece_of_brick"
    owner = np.array(getattr(sc, pieces)).copy()
    owner[corners] = sc.n_pieces
    setattr(sc, pieces, owner)
    sc.n_pieces += 1
    assert corners.sum() == 2
    vol = pkg.Volume(sc)
    glob = vol.moments_for(sc.views)
    vol.render_moments(sc.views, glob)
    ms, img = {}, {}
    for what, sel in (("piece", [sc.n_pieces - 1]), ("all", list(range(sc.n_pieces)))):
        mom, col = vol.moments_for(sc.views, len(sel)), pkg.Volume.color_buffer(sc.views, len(sel))
        best = 1e9
        for i in range(12):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            vol.render_moments(sc.views, mom, pieces=sel, mode=pkg.MBOIT_MOMENTS_PER_PIECE)
            vol.reconstruct_blend(sc.views, glob, col, pieces=sel, mode=pkg.MBOIT_COLOR_PER_PIECE)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b)) if i > 1 else best
        ms[what] = best
        n = len(sel)
        img[what] = (mom.view(n, -1)[-1], col.view(n, -1)[-1])
    for p, q in zip(img["piece"], img["all"]):
        assert torch.equal(p.view(torch.int32), q.view(torch.int32))
    assert (img["piece"][1] > 0).any()
    vol.close()
    assert ms["piece"] < 0.4 * ms["all"], ms
