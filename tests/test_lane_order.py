"""Two lanes of a warp that write the same shared memory: shuffles between them do not order their stores, a warp barrier does."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24695_b200", "csrc")


def test_denominators_go_behind_the_padding_they_are_written_over():
    """Heads of 112: the lane that holds chunk 6 of a row of the second box stores it turned, padding and all; then another lane of
    the warp stores the row's denominator there."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "umma_kernels.cu")).read())
    body = text[text.index("rope_apply_rows(uint8_t* sl"):text.index("apply_epilogue(uint32_t tmem_base")]
    turned = [m.start() for m in re.finditer(r"\*reinterpret_cast<uint4\*>\(c0 \+ HALF\) =", body)]
    denominator = [m.start() for m in re.finditer(r"\*reinterpret_cast<float\*>\(sl \+ HALF \+ row \* kRowBytes", body)]
    assert len(turned) == 1 and len(denominator) == 1 and turned[0] < denominator[0]
    between = body[turned[0]:denominator[0]]
    assert re.search(r"if \(D == 112\) __syncwarp\(\);", between)
    assert "}" not in between[between.index("__syncwarp"):]   # in the block of the denominator's store, so every lane comes to it
