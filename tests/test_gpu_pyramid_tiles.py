"""The level-0 copy and every coarser level are built from 64 x 32 pixel tiles in one
launch, the normals and gradients of a level in another.  Four levels at sizes around
the tile's edge (exact multiples, one pixel more or less, odd widths, whose rows are not
pair-aligned, and sizes smaller than a tile), with holes in the depth, each level against
the oracle at the tracked frame's last linearisation points.

Tolerances: those of the full-size comparison (validity per pixel exact outside the
margin pixels, the systems within the 1e-5 bar)."""
import copy

import pytest

from oracle import gn
from paper_2207_10940_gb300 import dri, synth
from parity import configs, new_stream
from test_gpu_fullsize import _check_level, _torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w, h, levels", [(128, 96, 4), (131, 97, 4), (127, 95, 3), (192, 129, 2), (257, 161, 4),
                                          (62, 46, 2)])
def test_levels(w, h, levels):
    _torch()
    seq = synth.frame_pair(seed=21, cam=synth.scaled_camera(w, h), dropout=0.02, trans_m=0.02)
    ocfg, dcfg = configs(seq, levels, (3, 3, 2, 2)[:levels])
    x_init = synth.initial_state(seq)
    st = new_stream(dcfg, x_init)
    dri.dri_push_imu(st.handle, seq.imu)
    dri.dri_upload_frame(st.handle, seq.frame_times[0], seq.depth[0], seq.intensity[0])
    assert dri.dri_track(st.handle).initialised == 1
    dri.dri_upload_frame(st.handle, seq.frame_times[1], seq.depth[1], seq.intensity[1])
    tr = gn.Tracker(ocfg, x_init)
    tr.push_imu(seq.imu)
    tr.track(seq.depth[0], seq.intensity[0], seq.frame_times[0])
    before = copy.deepcopy(tr)
    ores = tr.track(seq.depth[1], seq.intensity[1], seq.frame_times[1])
    for level in range(levels):
        x0, x1 = ores["points"][level]
        _check_level(st, before, seq, ocfg, level, x0, x1)
    st.close()
