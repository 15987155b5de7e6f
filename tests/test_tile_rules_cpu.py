"""What the launchers decide from the sizes of a call, without a GPU."""
import glob
import os
import re

from tile_rules import CSRC, rules, wt_cut


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


# us of linears on a B200 with tiles of 32, 64, .. 256 tokens (the first eight: 8-bit codes, the matmul alone)
MEASURED_CUTS = {
    (777, 3072, 1024): (12.4, 9.4, 8.9, 9.4, 8.4, 8.9, 9.3, 9.9),
    (1500, 3072, 256): (14.6, 10.8, 10.0, 9.1, 11.2, 11.8, 13.0, 8.8),
    (4096, 1024, 512): (14.6, 10.8, 10.1, 9.3, 11.3, 12.2, 13.0, 9.2),
    (900, 4096, 128): (12.9, 9.7, 9.5, 8.7, 10.9, 11.3, 12.5, 8.5),
    (200, 14336, 128): (11.4, 9.4, 9.0, 8.2, 11.0, 11.6, 8.0, 7.8),
    (2048, 8192, 1024): (54.2, 33.0, 29.8, 24.9, 30.6, 29.6, 32.2, 29.5),
    (8192, 4096, 128): (83.4, 51.4, 46.8, 39.2, 50.5, 47.5, 46.6, 43.6),
    (8192, 4096, 2048): (192.9, 102.3, 75.4, 61.1, 64.2, 59.1, 57.3, 54.3),
    (900, 4096, 1024): (19.4, 15.0, 14.6, 13.3, 15.4, 16.0, 17.2, 13.3),
    (600, 4096, 256): (11.6, 10.2, 9.7, 10.1, 8.4, 8.8, 9.2, 9.6),
    (2048, 8192, 256): (43.5, 29.1, 27.6, 23.6, 28.2, 27.6, 29.5, 27.6),
}


def test_tiles_of_the_kernel_for_one_byte_codes_are_near_the_best_measured():
    """Short rows too, where the epilogue and not the main loop sets the pace of a tile."""
    for (M, N, K), us in MEASURED_CUTS.items():
        cut = wt_cut(M, N, K)
        assert not cut.shared and us[cut.tokens // 32 - 1] <= 1.06 * min(us), ((M, N, K), cut)
