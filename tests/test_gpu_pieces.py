"""Per-piece images from one march per ray against each piece's own march
(a list of one piece takes that one): the same bits for every volume kind,
moment set, step and list of pieces."""
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


def _grid(n, views):
    sc = scenes.blobs512(width=views[0][0], height=views[0][1], n_pieces=9, n=n)
    sc.views += [scenes.ortho_view(sc.field.shape[::-1], (-0.3, 0.8, 0.4), w, h) for w, h in views[1:]]
    return sc


def _octree(adaptive=False, holes=False):
    sc = scenes.amr_blobs(base=4, max_level=2, width=45, height=38, n_pieces=9)
    sc.adaptive_step = adaptive
    if holes:
        keep = np.arange(len(sc.leaves)) % 11 != 3
        sc.leaves, sc.values, sc.piece_of_leaf = sc.leaves[keep], sc.values[keep], sc.piece_of_leaf[keep]
    return sc


SCENES = {
    "grid_vec": lambda: _grid(64, [(50, 41), (33, 20)]),       # 16-byte rows; two views, a ragged plane
    "grid_odd": lambda: _grid(51, [(37, 29)]),                  # no 16-byte rows
    "octree": _octree,
    "octree_adaptive": lambda: _octree(adaptive=True),
    "octree_holes": lambda: _octree(holes=True),
    "mesh": lambda: scenes.tet_mesh(n=12, n_pieces=9, width=40, height=35),
}
SETS = [("power4", "f32", 5e-5), ("power6", "f32", 1e-3), ("power8", "f32", 1e-3), ("trig6", "bf16", 2e-2),
        ("trig8", "f16", 2e-3)]


def _images(pkg, vol, sc, pieces, glob):
    """(per-piece moments, per-piece colours) of the listed pieces, buffers filled with rubbish first."""
    n = len(pieces)
    mom = vol.moments_for(sc.views, n)
    mom.fill_(7.0)
    col = pkg.Volume.color_buffer(sc.views, n).fill_(7.0)
    vol.render_moments(sc.views, mom, pieces=pieces, mode=pkg.MBOIT_MOMENTS_PER_PIECE)
    n1 = vol.stats()["samples_pass1"]
    vol.reconstruct_blend(sc.views, glob, col, pieces=pieces, mode=pkg.MBOIT_COLOR_PER_PIECE)
    st = vol.stats()
    vol.synchronize()
    words = [pkg.mboit_moment_image_bytes(v.width, v.height, vol.moment_set, vol.storage) // 4 for v in sc.views]
    m, c, out = 0, 0, []
    for v, w in zip(sc.views, words):
        P = (v.width * v.height + 3) // 4 * 4
        slabs = mom[m:m + n * w].view(n, w)
        # the words past the last pixel of each plane are not part of the image
        b0, rest = slabs[:, :P][:, :v.width * v.height], slabs[:, P:]
        if vol.moment_set in (pkg.MBOIT_TRIG6, pkg.MBOIT_TRIG8):
            rest = rest.reshape(n, -1, P)[:, :, :v.width * v.height]
        else:
            first = rest[:, :4 * P].reshape(n, P, 4)[:, :v.width * v.height].flatten(1)
            tail = rest[:, 4 * P:]
            rest = first if not tail.shape[1] else \
                __import__("torch").cat([first, tail.reshape(n, P, -1)[:, :v.width * v.height].flatten(1)], 1)
        out.append((b0.clone(), rest.clone(), col[c:c + n * 4 * v.width * v.height].view(n, -1).clone()))
        m += n * w
        c += n * 4 * v.width * v.height
    return out, n1, st["samples_pass2"]


@pytest.mark.parametrize("ms, storage, bias", SETS)
@pytest.mark.parametrize("name", list(SCENES))
def test_one_march_equals_own_marches(pkg, name, ms, storage, bias):
    import torch
    sc = SCENES[name]()
    sc.moment_set, sc.storage, sc.moment_bias = ms, storage, bias
    vol = pkg.Volume(sc)
    glob = vol.moments_for(sc.views)
    vol.render_moments(sc.views, glob)
    own = [_images(pkg, vol, sc, [p], glob) for p in range(sc.n_pieces)]
    # every piece in order; a partial list in another order; a piece named twice
    lists = [list(range(sc.n_pieces)), [7, 0, 4, 2, 8, 1, 6], [3, 5, 3, 0, 1, 2, 4, 6, 7, 8]]
    for pieces in lists:
        got, n1, n2 = _images(pkg, vol, sc, pieces, glob)
        for vi in range(len(sc.views)):
            for j, p in enumerate(pieces):
                for a, b in zip(got[vi], own[p][0][vi]):
                    assert torch.equal(a[j].contiguous().view(torch.int32), b[0].contiguous().view(torch.int32))
        assert n1 == sum(own[p][1] for p in pieces)
        assert n2 == sum(own[p][2] for p in pieces)
    vol.close()
