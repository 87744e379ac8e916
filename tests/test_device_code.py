"""Rules of the CUDA sources that no run on one GPU can show broken: convergence before warp-aligned
instructions, and launch attributes on every device."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_04929_gb300", "csrc")


def sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            yield os.path.basename(path), f.read()


def test_cluster_barriers_follow_a_warp_reconvergence():
    """barrier.cluster.*.aligned must be executed by all threads of a warp together, which nothing
    but an explicit __syncwarp() guarantees after a branch that lanes took apart."""
    found = 0
    for name, text in sources():
        for m in re.finditer(r"asm volatile\(\s*\"barrier\.cluster\.arrive[^\"]*\.aligned", text):
            before = re.sub(r"//[^\n]*", "", text[:m.start()]).rstrip()
            assert before.endswith("__syncwarp();"), (name, text[m.start() - 200:m.end()])
            found += 1
    assert found >= 1


def test_launch_attributes_are_set_on_every_device():
    """cudaFuncSetAttribute acts on the current device only; a flag kept by the process would leave a context
    on another device without it, and is written by several host threads at once."""
    for name, text in sources():
        text = re.sub(r"//[^\n]*", "", text)
        flags = [m.group(0) for m in re.finditer(r"\bstatic\s+(?!constexpr|const\b)(?:bool|int|std::once_flag|std::atomic<\w+>)\s+\w+\s*(?:=|;|\{)", text)]
        assert not flags, (name, flags)
