"""What the launchers decide from the sizes of a call, without a GPU."""
import glob
import os
import re

from tile_rules import CSRC, rules


def test_widths_of_cta_pair_tiles_are_shapes_of_the_instruction():
    """An 8-bit integer matrix instruction of two CTAs is specified for multiples of 32 columns; 208 and 240 are not."""
    R = rules()
    assert [n for n in range(1, 300) if R.mma_width(n)] == list(range(32, 257, 32))
    widths = {R.pair_width(M, N, pairs) for pairs in (74, 66, 1) for M in (1, 65, 200, 256, 257, 1003, 2048, 4096, 8192)
              for N in list(range(8, 4096, 88)) + list(range(4096, 70000, 1000)) + [74 * w for w in range(200, 260)]}
    assert len(widths) > 1 and all(R.mma_width(n) for n in widths), widths


def test_widths_of_cta_pair_instructions_in_the_source():
    """Whoever builds the instruction descriptor of a CTA pair (256 rows) checks the width where it is known."""
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = open(path).read()
        if re.search(r"umma_idesc_i8\((TM|RT|kPair)", text):
            assert "umma_i8_pair_width(" in text, path
