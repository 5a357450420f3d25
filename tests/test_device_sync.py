"""Rules of synchronisation that the device code keeps by construction, read from its
source (a break of one of them is a matter of timing and seldom shows in results)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_10940_gb300", "csrc")


def sources():
    """Device sources by file name, without their comments."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        yield os.path.basename(path), re.sub(r"//[^\n]*", "", open(path).read())


def test_hand_off_barriers_have_an_id_of_their_own():
    """A warp that only arrives on a named barrier may reach a second use of it before
    the warps that wait have passed the first; the barrier then counts it twice and
    opens without one of them.  So a barrier with a bar_arrive serves that one
    hand-off: one arriving and one waiting place, of the same thread count."""
    found = 0
    for name, text in sources():
        arrive, sync = {}, {}
        for kind, bid, n in re.findall(r"\bbar_(arrive|sync)<(\d+), (\d+)>\(\)", text):
            (arrive if kind == "arrive" else sync).setdefault(int(bid), []).append(int(n))
        for bid, counts in arrive.items():
            found += 1
            assert len(counts) == 1 and sync.get(bid) == counts, (name, bid, counts, sync.get(bid))
    assert found >= 4


def test_a_block_that_shares_its_launch_with_the_step_decides_as_one():
    """The block that assembles the last system reads the camera's status, which the
    step's block of the same launch may be writing: its threads must not each decide by
    what they happened to read (the code behind the test has block barriers)."""
    text = dict(sources())["solve.cu"]
    body = text[text.index("void step_lin_block("):]
    body = body[:body.index("\n}")]
    tests = re.findall(r"if \(([^;]*)\) return;", body)
    assert any("status" in t for t in tests)
    assert all(t.startswith("__syncthreads_or(") for t in tests if "status" in t), tests


def test_shuffle_masks_are_not_taken_from_the_running_threads():
    """__activemask() names the threads that happen to run together, which need not be
    all that a branch holds; a mask for the branch is taken by a ballot before it."""
    for name, text in sources():
        assert "__activemask" not in text, name
