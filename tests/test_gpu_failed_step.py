"""A frame whose only iteration fails: the frame's last launch runs the step and, in a
second block per camera, the system for the marginalisation, and the step's failure is
written while that block may be reading it.  Cameras of a batch in turn get a prior that
makes the step fail (a negative pose information, which the step's pivots refuse): those
frames are lost, state and reference stay, the other cameras' frames and, with their own
prior back, the lost cameras' next frames give the same bits as without the failure."""
import numpy as np
import pytest

from paper_2207_10940_gb300 import dri, synth
from parity import configs

pytestmark = pytest.mark.gpu

N = 40                                  # 20 failing beside 20 that go on: 80 blocks in the last launch


def _streams(torch, seq):
    _, dcfg = configs(seq, 1, (1,))
    x_init = synth.initial_state(seq)
    ts = torch.cuda.Stream()
    sts = [dri.Stream(dcfg, dri.state_from_dict(x_init, x_init.get("t", 0.0)), ts) for _ in range(N)]
    for st in sts:
        dri.dri_push_imu(st.handle, seq.imu)
    return sts


def _frame(sts, seq, i):
    for st in sts:
        dri.dri_upload_frame(st.handle, seq.frame_times[i], seq.depth[i], seq.intensity[i])
    return [r.status for r in dri.dri_track_batch(sts)]


def _states(sts):
    return [dri.dri_get_state(st.handle, with_prior=True) for st in sts]


def _set(st, state, information=0.0):
    """Sets the state with its prior, `information` added on the pose; returns it as
    stored (the quaternions are normalised again)."""
    x, H, b = state
    Hp = H.copy()
    Hp[:6, :6] += information * np.eye(6)
    dri.dri_set_state(st.handle, x, Hp, b)
    return dri.dri_get_state(st.handle), H, b


def _run(torch, seq, failing, frame_1):
    """States of N equal cameras after frame 1 (not given to them unless frame_1) and
    after frame 2; the failing ones' prior is replaced for frame 1 and put back."""
    sts = _streams(torch, seq)
    assert _frame(sts, seq, 0) == [0] * N
    kept = {k: _set(sts[k], dri.dri_get_state(sts[k].handle, with_prior=True), -1e15 if frame_1 else 0.0)
            for k in failing}
    if frame_1:
        assert _frame(sts, seq, 1) == [dri.DRI_ELOST if k in kept else 0 for k in range(N)]
    first = _states(sts)
    for k, state in kept.items():
        assert bytes(first[k][0]) == bytes(state[0])
        _set(sts[k], state)
    assert _frame(sts, seq, 2) == [0] * N
    second = _states(sts)
    for st in sts:
        st.close()
    return first, second


def _same(a, b):
    return bytes(a[0]) == bytes(b[0]) and np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])


def test_failed_last_step_leaves_the_others_and_the_next_frame():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    seq = synth.sinusoid_sequence(seed=14, cam=synth.scaled_camera(96, 72), n_frames=3)
    failing = range(0, N, 2)
    good = _run(torch, seq, [], True)
    mixed = _run(torch, seq, failing, True)
    skipped = _run(torch, seq, failing, False)
    for k in range(N):
        if k in failing:
            assert _same(mixed[1][k], skipped[1][k])
        else:
            assert _same(mixed[0][k], good[0][k]) and _same(mixed[1][k], good[1][k])
