"""The allocation-free pair entry reports as many margin decisions as its own per-pixel
flags mark: its last block reads the counts that every warp of every block has added to,
so each warp's addition must be visible before its block counts as done.  Exact (integer
counts), at the entry's smallest size (two blocks), a ragged one and its largest."""
import ctypes

import pytest

from oracle.so3 import State
from paper_2207_10940_gb300 import dri, synth
from parity import configs, to_dri

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [{}, {"occlusion_thr": 0.05, "icp_depth_weight": 1}, {"precision_flags": 3}],
                         ids=["default", "options", "fp16"])
@pytest.mark.parametrize("w, h", [(8, 8), (131, 97), (320, 240)])
def test_margin_counts_equal_the_flags(w, h, opts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    seq = synth.frame_pair(seed=3, cam=synth.scaled_camera(w, h), dropout=0.02)
    _, dcfg = configs(seq, 1, (3,), **opts)
    images = [torch.from_numpy(a).cuda() for a in (seq.depth[0], seq.intensity[0], seq.depth[1], seq.intensity[1])]
    out = torch.zeros(ctypes.sizeof(dri.dri_linearisation), dtype=torch.uint8, device="cuda")
    flags = torch.zeros(w * h, dtype=torch.uint8, device="cuda")
    # at one common pose, where border pixels project onto the image's bound, and at the
    # two true ones
    first = to_dri(State.from_dict(synth.initial_state(seq)))
    for x0, x1 in ((first, first), tuple(to_dri(State.from_dict(g)) for g in seq.gt)):
        for _ in range(20):
            dri.dri_linearise_pair_noalloc(dcfg, *images, first, x0, x1, out, flags, torch.cuda.current_stream())
            got = dri.dri_linearisation.from_buffer_copy(out.cpu().numpy().tobytes())
            marks = flags.cpu()
            assert got.n_margin_icp == int(((marks & 64) != 0).sum())
            assert got.n_margin_rgb == int(((marks & 128) != 0).sum())
