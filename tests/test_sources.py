"""Rules of the CUDA sources that no run can show to be kept (a breach may go well on one GPU for years)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2303_08365_gb300", "csrc")


def statements(path):
    """The file's statements without comments, blanks folded."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path, encoding="utf-8").read(), flags=re.S)
    return [" ".join(s.split()) for s in re.split(r"[;{}]", text)]


def test_a_vote_on_waits_is_followed_by_a_warp_barrier():
    """Lanes that acquire different words pass what they have acquired on to each other by __syncwarp:
    __all_sync alone orders no memory."""
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = statements(path)
        for k, s in enumerate(code):
            if re.search(r"__all_sync\(0xffffffffu, ok\)", s):
                seen += 1
                assert code[k + 1] == "__syncwarp()", (os.path.basename(path), s)
    assert seen >= 2


def test_the_fma_chain_reads_its_weights_by_plain_loads():
    """wide_chain's weights may lie among a kernel's parameters (a single grid's tile kernel):
    __ldg is a load from global memory and undefined there."""
    code = statements(os.path.join(CSRC, "wide.cuh"))
    at = next(k for k, s in enumerate(code) if re.search(r"double wide_chain\(", s))
    body = code[at + 1:code.index("return acc", at)]
    assert any("fma(wdev[k], v[k], acc)" in s for s in body)
    assert not any("__ldg" in s for s in body)
