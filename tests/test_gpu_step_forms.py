"""The two forms of the Gauss-Newton step: the covariance form (every iteration
but a frame's last) takes up to 64 IMU pieces per frame and needs the prior to
inform every non-pose component; otherwise a frame's steps all run in the
information form.  Both against the oracle at the edges of that choice: 1, 2,
64 and 65 pieces (the tree of pre-integrations: a single leaf, one pair, full,
one beyond), and a prior without information on the gyro bias.

Tolerances: the pose bar of the library; the non-pose state within 10% of a
standard deviation of the oracle's H* (the systems' 1e-5 bar leaves ~0.03)."""
import numpy as np
import pytest

from oracle import gn
from oracle.so3 import boxminus
from paper_2207_10940_gb300 import dri, synth
from parity import POSE_M, POSE_RAD, configs, new_stream, pose_error, to_oracle

pytestmark = pytest.mark.gpu


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _check(res, ores):
    da, dr = pose_error(res.x1, ores["x1"])
    assert da < POSE_RAD and dr < POSE_M, (da, dr)
    d = boxminus(to_oracle(res.x1), ores["x1"])
    assert float(np.sqrt(d @ ores["H_prior"] @ d)) < 0.1


# A single piece gives the nine position, rotation and velocity rows a covariance
# of rank six: only the gyro-only variant, which weighs the rotation rows alone,
# can track with it.
@pytest.mark.parametrize("mode, rate", [(dri.DRI_TRACK_GYRO_ONLY, 30.0)] + [
    (m, r) for m in (dri.DRI_TRACK_INERTIAL, dri.DRI_TRACK_GYRO_ONLY) for r in (60.0, 1920.0, 1950.0)])
def test_pieces(mode, rate):
    _torch()
    seq = synth.sinusoid_sequence(seed=12, cam=synth.scaled_camera(160, 120), n_frames=2, rate=rate)
    ocfg, dcfg = configs(seq, 2, (6, 4), track_mode=mode)
    x_init = synth.initial_state(seq)
    st = new_stream(dcfg, x_init)
    dri.dri_push_imu(st.handle, seq.imu)
    tr = gn.Tracker(ocfg, x_init)
    tr.push_imu(seq.imu)
    for i in range(2):
        dri.dri_upload_frame(st.handle, seq.frame_times[i], seq.depth[i], seq.intensity[i])
        res = dri.dri_track(st.handle)
        assert res.status == 0
        ores = tr.track(seq.depth[i], seq.intensity[i], seq.frame_times[i])
    st.close()
    _check(res, ores)


def test_prior_without_gyro_bias_information():
    _torch()
    seq = synth.sinusoid_sequence(seed=13, cam=synth.scaled_camera(160, 120), n_frames=2)
    ocfg, dcfg = configs(seq, 2, (6, 4))
    x_init = synth.initial_state(seq)
    st = new_stream(dcfg, x_init)
    dri.dri_push_imu(st.handle, seq.imu)
    tr = gn.Tracker(ocfg, x_init)
    tr.push_imu(seq.imu)
    dri.dri_upload_frame(st.handle, seq.frame_times[0], seq.depth[0], seq.intensity[0])
    assert dri.dri_track(st.handle).initialised == 1
    tr.track(seq.depth[0], seq.intensity[0], seq.frame_times[0])
    x, H, b = dri.dri_get_state(st.handle, with_prior=True)
    H[9:12, 9:12] = 0.0
    dri.dri_set_state(st.handle, x, H, b)
    tr.Hs = H.copy()
    dri.dri_upload_frame(st.handle, seq.frame_times[1], seq.depth[1], seq.intensity[1])
    res = dri.dri_track(st.handle)
    assert res.status == 0
    ores = tr.track(seq.depth[1], seq.intensity[1], seq.frame_times[1])
    st.close()
    _check(res, ores)
