"""What can be told from the kernels' sources alone, without a GPU."""
import glob
import os
import re

DEVICE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_13585_b200", "csrc", "device")


def _sources():
    out = {}
    for f in sorted(glob.glob(os.path.join(DEVICE, "*.cuh"))):
        out[os.path.basename(f)] = re.sub(r"//[^\n]*", "", open(f).read())
    return out


def _block_behind(text, at):
    """The text between the first brace behind `at` and the brace that closes it."""
    at = text.index("{", at)
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at + 1:i]
    raise AssertionError("unbalanced braces")


def test_shared_memory_of_another_block_is_written_between_two_barriers():
    """All blocks of a cluster must be known to have started before one writes to another's shared memory, and to have written
    before it is read.  Only FirstBlock writes there, with what its wait for the start returns, and every kernel that is launched
    as a cluster arrives with its first statement, waits before it writes and waits again before it reads."""
    sources = _sources()
    remote = r"mapa\.|(?:st|ld|atom|red)(?:\.\w+)*\.shared::cluster|barrier\.cluster"
    clusters = 0
    for name, text in sources.items():
        if name == "skeletons.cuh":
            at = text.index("class FirstBlock")
            first_block = _block_behind(text, at)
            opened = _block_behind(first_block, first_block.index("class Open"))
            assert "mapa" in opened and "st.shared::cluster" in opened and "barrier.cluster.arrive.release" in opened
            assert re.search(r"private:\s*friend class FirstBlock;\s*__device__ __forceinline__ Open\(\)", opened)
            outside = first_block.replace(opened, "")
            assert outside.index("barrier.cluster.arrive.relaxed") < outside.index("barrier.cluster.wait.acquire") < outside.index("return Open()")
            text = text.replace(first_block, "")
        assert not re.search(remote, text), name
        for m in re.finditer(r"__cluster_dims__", text):
            body = _block_behind(text, m.start())
            assert body.strip().startswith("const FirstBlock first;"), name
            steps = ["first.all_have_started()", "open.put(", "open.all_have_written()"]
            assert [body.count(s) for s in steps] == [1, 1, 1], name
            assert sorted(steps, key=body.index) == steps, name
            # (nobody leaves before the last of them)
            assert "return" not in re.sub(r"\[[^\]]*\]\(auto ic\)", "", body[:body.index(steps[2])]), name
            clusters += 1
    assert clusters == 2
