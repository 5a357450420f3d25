"""The RGB-D-only step solves its 6 x 6 system to FP64 rounding: one iteration from the
identity pose against the system of the same pixel sums (dri_linearise at that pose; the
last iteration counts margins, as dri_linearise does, so both run one kernel), residual in
exact arithmetic.

Tolerance: with d_i = sqrt(H_ii), |H| <= d d^T, and an LDL^T solution of order 6 takes
about 50 roundings on any entry's way (19 of the factorisation and the substitutions, as
many for products with a reciprocal, the rest for the sum of the two terms' systems and
reading the step off the pose).  They are independent: sqrt(50) u = 7.9e-16 is the scaled
residual's standard size, and two and a half times that, 2e-15, the bar for the largest of
the six rows of 32 systems."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2207_10940_gb300 import dri, synth
from parity import configs, new_stream

pytestmark = pytest.mark.gpu

BAR = 2e-15


def _rotation_vector(q):
    v = np.array(q[1:])
    n = np.linalg.norm(v)
    return 2.0 * np.arctan2(n, q[0]) / n * v


def test_step_solves_its_system_to_rounding():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    worst = []
    for seed in range(32):
        seq = synth.frame_pair(seed=100 + seed, cam=synth.scaled_camera(96, 72))
        _, dcfg = configs(seq, 1, (1,), track_mode=dri.DRI_TRACK_RGBD_ONLY)
        dcfg.count_margins = 1
        x_init = synth.initial_state(seq)
        assert not np.any(x_init["r_WC"]) and list(x_init["q_WC"]) == [1.0, 0.0, 0.0, 0.0]
        st = new_stream(dcfg, x_init)
        dri.dri_push_imu(st.handle, seq.imu)
        dri.dri_upload_frame(st.handle, seq.frame_times[0], seq.depth[0], seq.intensity[0])
        assert dri.dri_track(st.handle).initialised == 1
        dri.dri_upload_frame(st.handle, seq.frame_times[1], seq.depth[1], seq.intensity[1])
        x = dri.dri_get_state(st.handle)
        out, _ = dri.dri_linearise(st.handle, 0, x, x)
        res = dri.dri_track(st.handle)
        assert res.status == 0
        st.close()
        assert res.n_icp[0] == out.n_icp and res.n_rgb[0] == out.n_rgb
        dx = np.concatenate([list(res.x1.r_WC), _rotation_vector(list(res.x1.q_WC))])
        H = [[Fraction(out.H_icp[6 * i + j]) + Fraction(out.H_rgb[6 * i + j]) for j in range(6)] for i in range(6)]
        b = [Fraction(out.b_icp[i]) + Fraction(out.b_rgb[i]) for i in range(6)]
        d = np.array([float(H[i][i]) ** 0.5 for i in range(6)])
        r = np.array([float(b[i] - sum(H[i][j] * Fraction(dx[j]) for j in range(6))) for i in range(6)])
        worst.append(float(np.max(np.abs(r) / (d * float(d @ np.abs(dx))))))
    assert max(worst) < BAR, sorted(worst)[-5:]
