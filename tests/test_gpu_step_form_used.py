"""Which form of the Gauss-Newton step a frame runs in: the covariance form for up to 64
IMU pieces and a prior that informs every non-pose component, the information form
otherwise (both meet the same tolerances, so results alone do not tell).  Read from the
stream's control record in its workspace, at the offsets that the C++ compiler gives:
the frame's pieces and `lin_split`, which only a last step in covariance form sets."""
import os
import shutil
import struct
import subprocess

import pytest

from paper_2207_10940_gb300 import build, dri, synth
from parity import configs, new_stream

pytestmark = pytest.mark.gpu

PROGRAM = """#include <cstdio>
#define __ldg(p) (*(p))
#include "dri_internal.h"
int main() { std::printf("%zu %zu", offsetof(dri::Ctrl, elim.np), offsetof(dri::Ctrl, lin_split)); }
"""


@pytest.fixture(scope="module")
def record(tmp_path_factory):
    """Function of a stream: (pieces, lin_split) of its last frame."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("ctrl")
    (d / "offsets.cpp").write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    subprocess.run([shutil.which("g++"), "-std=c++17", "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"),
                    "-I", cuda, "-o", str(d / "offsets"), str(d / "offsets.cpp")], check=True)
    offsets = [int(v) for v in subprocess.run([str(d / "offsets")], capture_output=True, check=True).stdout.split()]

    def read(st):
        torch.cuda.synchronize()
        base = -st.workspace.data_ptr() % 256          # the record is the workspace's first part
        return tuple(struct.unpack("i", st.workspace[base + o:base + o + 4].cpu().numpy().tobytes())[0]
                     for o in offsets)
    return read


def _track(seq, mode=dri.DRI_TRACK_INERTIAL, without_gyro_bias=False):
    _, dcfg = configs(seq, 2, (6, 4), track_mode=mode)
    st = new_stream(dcfg, synth.initial_state(seq))
    dri.dri_push_imu(st.handle, seq.imu)
    for i in range(2):
        if i and without_gyro_bias:
            x, H, b = dri.dri_get_state(st.handle, with_prior=True)
            H[9:12, 9:12] = 0.0
            dri.dri_set_state(st.handle, x, H, b)
        dri.dri_upload_frame(st.handle, seq.frame_times[i], seq.depth[i], seq.intensity[i])
        assert dri.dri_track(st.handle).status == 0
    return st


# the cases of the comparison with the oracle (test_gpu_step_forms.py)
@pytest.mark.parametrize("mode, rate, pieces", [(dri.DRI_TRACK_GYRO_ONLY, 30.0, 1)] + [
    (m, r, n) for m in (dri.DRI_TRACK_INERTIAL, dri.DRI_TRACK_GYRO_ONLY)
    for r, n in ((60.0, 2), (1920.0, 64), (1950.0, 65))])
def test_form_by_pieces(record, mode, rate, pieces):
    seq = synth.sinusoid_sequence(seed=12, cam=synth.scaled_camera(160, 120), n_frames=2, rate=rate)
    st = _track(seq, mode)
    assert record(st) == (pieces, int(pieces <= 64))
    st.close()


def test_form_without_gyro_bias_information(record):
    seq = synth.sinusoid_sequence(seed=13, cam=synth.scaled_camera(160, 120), n_frames=2)
    st = _track(seq, without_gyro_bias=True)
    assert record(st)[1] == 0
    st.close()
