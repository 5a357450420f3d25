"""A prior given by its upper triangle (dri_set_state): every form of the step and the
marginalisation take H* from there, so the frame's first step is that of the full symmetric
matrix.  A dense prior of a tracked frame, one iteration; the states agree to 1e-6 of a
standard deviation of the prior (the linearisation point is the prior's mean up to 1e-16,
so the triangle that only the prior's gradient reads contributes rounding)."""
import numpy as np
import pytest

from oracle.so3 import boxminus
from paper_2207_10940_gb300 import dri, synth
from parity import configs, new_stream, to_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [dri.DRI_TRACK_INERTIAL, dri.DRI_TRACK_GYRO_ONLY])
def test_upper_triangle_is_enough(mode):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    seq = synth.sinusoid_sequence(seed=15, cam=synth.scaled_camera(96, 72), n_frames=3)
    _, dcfg = configs(seq, 1, (1,), track_mode=mode)
    x_init = synth.initial_state(seq)
    got = []
    for part in (lambda H: H, np.triu):
        st = new_stream(dcfg, x_init)
        dri.dri_push_imu(st.handle, seq.imu)
        for i in range(3):
            if i == 2:
                x, H, b = dri.dri_get_state(st.handle, with_prior=True)
                assert np.array_equal(H, H.T) and np.count_nonzero(np.triu(H, 1)) > 10
                dri.dri_set_state(st.handle, x, part(H), b)
            dri.dri_upload_frame(st.handle, seq.frame_times[i], seq.depth[i], seq.intensity[i])
            assert dri.dri_track(st.handle).status == 0
        got.append((dri.dri_get_state(st.handle, with_prior=True)))
        st.close()
    (xa, Ha, ba), (xb, Hb, bb) = got
    d = boxminus(to_oracle(xa), to_oracle(xb))
    assert float(np.sqrt(abs(d @ Ha @ d))) < 1e-6
    s = np.sqrt(np.diag(Ha)) + 1e-300
    assert np.all(np.abs(Ha - Hb) <= 1e-6 * np.outer(s, s))
