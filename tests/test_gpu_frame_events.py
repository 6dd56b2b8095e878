"""What the frame's events enclose: pass 1's time holds the check of the index
tables.  An octree of 2048 finest cells a side has 256^3 finest bricks, 134 MB
of map and words to check; a view that misses the domain leaves pass 1 nothing
else to do.  Reading 134 MB at 27 TB/s (more than three times the nominal
memory rate, so above what the L2 can add) takes 5 us, so pass 1 takes at
least that much longer than on an octree with a map of 8 entries."""
import statistics

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


@pytest.mark.parametrize("launches", [1, 2])
def test_pass1_time_holds_the_table_check(pkg, launches):
    f = np.float32
    # an orthographic view along z, beside the domain
    view = scenes.View(np.array([-9e3, -9e3, -1e3], f), np.array([1, 0, 0], f), np.array([0, 1, 0], f),
                       np.array([0, 0, 1], f), 32, 32, scenes.ORTHO, f(100), f(100), f(1), f(5e3))
    ms = []
    for level in (0, 7):
        sc = scenes.amr_blobs(base=2, max_level=level, width=8, height=8, n_pieces=2, alpha_max=0.05)
        vol = pkg.Volume(sc)
        vol.set_frame_launches(launches)
        mom, col = vol.moments_for([view]), pkg.Volume.color_buffer([view])
        t = []
        for _ in range(15):
            vol.render_frame([view], mom, col)
            t.append(vol.stats()["frame_pass1_ms"])
        assert vol.stats()["samples_pass1"] == 0
        ms.append(statistics.median(t[5:]))
        vol.close()
    assert ms[1] - ms[0] >= 5e-3, ms
