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


def test_low_rank_factor_blocks_end_after_their_last_read():
    """k_big_lr reads a block's rows in chunks of LNC columns, past the row's end in the last chunk; the block's
    size (as the source computes it) covers the last row's reads, so that none falls into a block that the
    same product writes."""
    text = dict(sources())["k_big_lr.cu"]
    lnc = int(re.search(r"constexpr int LNC = (\d+);", text).group(1))
    block = re.search(r"const size_t blk = ([^;]+);", text).group(1)
    body = re.search(r"size_t lr_block\(int d, int ldw\) \{ return ([^;]+); \}", text)
    expr = (body.group(1) if body else block).replace("(size_t)", "")
    for d in (1, 69, 154, 512):
        for w in range(1, 65):
            ldw = (w + 1) & ~1
            ldw += 2 if (ldw >> 1) & 1 == 0 else 0
            last = (d - 1) * ldw + (w - 1) // lnc * lnc + lnc - 1
            assert last < eval(expr, {"d": d, "ldw": ldw, "LNC": lnc}), (d, w)
            assert eval(expr, {"d": d, "ldw": ldw, "LNC": lnc}) % 2 == 0      # the next block's 16-byte loads
