"""A frame interval covered by one IMU sample (samples as often as frames): its noise has
six components, the covariance of the nine position, rotation and velocity rows has rank
six, and Sigma^-1 does not exist.  Such a frame is lost whatever its pivots round to, the
state stays, and the next frame, two samples on, tracks."""
import pytest

from paper_2207_10940_gb300 import dri, synth
from parity import configs, new_stream

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rate", [30.0, 60.0])
@pytest.mark.parametrize("kw", [{}, {"imu_mode": dri.DRI_IMU_FIRST_ORDER}, {"gravity_dof": dri.DRI_GRAVITY_3D}],
                         ids=["default", "first-order", "3-D gravity"])
def test_single_piece_is_lost_and_the_next_frame_tracks(rate, kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for seed in range(16):
        seq = synth.sinusoid_sequence(seed=40 + seed, cam=synth.scaled_camera(96, 72), n_frames=3, fps=rate, rate=rate)
        _, dcfg = configs(seq, 2, (4, 3))
        for k, v in kw.items():
            setattr(dcfg, k, v)
        st = new_stream(dcfg, synth.initial_state(seq))
        dri.dri_push_imu(st.handle, seq.imu)
        status = []
        for i in range(3):
            dri.dri_upload_frame(st.handle, seq.frame_times[i], seq.depth[i], seq.intensity[i])
            before = dri.dri_get_state(st.handle) if i else None
            status.append(dri.dri_track(st.handle).status)
            if i == 1:
                assert bytes(dri.dri_get_state(st.handle)) == bytes(before), seed
        st.close()
        assert status == [0, dri.DRI_ELOST, 0], (seed, status)
