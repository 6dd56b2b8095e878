"""Grids nobody has tuned (the views choose the windows), windows of selections,
and repeated multi-volume frames: the same bits as configuration 0 and as
each volume's own frame."""
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


def _render(pkg, vol, views, pieces):
    out = []
    for call in ("frame", "split"):
        mom, col = vol.moments_for(views), pkg.Volume.color_buffer(views)
        if call == "frame":
            vol.render_frame(views, mom, col)
        else:
            vol.render_moments(views, mom, pieces=pieces)
            vol.reconstruct_blend(views, mom, col, pieces=pieces)
        vol.synchronize()
        out += [mom.clone(), col.clone()]
    return out


@pytest.mark.parametrize("n, size, chosen", [(64, (200, 160), 6), (64, (20, 24), 0), (51, (150, 111), 0)])
@pytest.mark.parametrize("unowned", [False, True])
def test_windows_nobody_chose(pkg, n, size, chosen, unowned):
    import torch
    sc = scenes.blobs512(width=size[0], height=size[1], n_pieces=6, n=n)
    if unowned:   # a piece that no volume owns: the frames select too
        sc.piece_of_brick = np.where(sc.piece_of_brick == 5, -1, sc.piece_of_brick)
        sc.n_pieces = 5
    pieces = [0, 2, 3]
    vol = pkg.Volume(sc)
    got = _render(pkg, vol, sc.views, pieces)
    assert vol.stats()["tuning_pass1"] == chosen
    for cfg in (0, 3):
        if cfg and n % 4:
            continue
        vol.set_tuning(cfg, cfg)
        for a, b in zip(got, _render(pkg, vol, sc.views, pieces)):
            assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    vol.close()


def test_repeated_multi_frames(pkg):
    """The cache rows of the last views are kept: other views, and the first
    again, must each get their own count."""
    import torch
    vols = [pkg.Volume(scenes.blobs64(n_pieces=3, seed=1001)) for _ in range(2)]
    views = {s: [scenes.ortho_view((64, 64, 64), (0.5, 0.3 + 0.2 * i, 0.7), s, s + 3) for i in range(3)]
             for s in (24, 90, 41)}
    own = {}
    for s, vw in views.items():
        for i, v in enumerate(vw):
            mom, col = pkg.Volume.moment_buffer([v]), pkg.Volume.color_buffer([v])
            vols[i % 2].render_frame([v], mom, col)
            vols[i % 2].synchronize()
            own[s, i] = col.clone()
    for s in (24, 24, 90, 90, 41, 24):
        mom, col = pkg.Volume.moment_buffer(views[s]), pkg.Volume.color_buffer(views[s])
        pkg.Volume.render_frame_multi(vols, views[s], [0, 1, 0], mom, col)
        vols[0].synchronize()
        for i, c in enumerate(col.view(3, -1)):
            assert torch.equal(c, own[s, i])
    for v in vols:
        v.close()
