"""What the launchers decide from the sizes of a call, without a GPU."""
import glob
import os
import re

from tile_rules import CSRC, rules, wt_ahead, wt_cut


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


# us of linears (quantise pass included) with packed codes and with codes of one byte
MEASURED_SIDES = {
    (65, 8, 256): (4.9, 5.8), (65, 14336, 4096): (19.5, 13.3), (100, 14336, 2048): (15.1, 10.9),
    (129, 72, 14336): (48.3, 16.6), (256, 14336, 256): (9.5, 10.2), (333, 6144, 2048): (15.3, 11.9),
    (333, 14336, 8192): (48.8, 39.8), (400, 1024, 512): (9.7, 6.6), (400, 8192, 256): (9.6, 10.3),
    (512, 64, 256): (5.8, 5.9), (512, 128, 4096): (20.2, 10.7), (600, 1024, 256): (8.9, 7.1),
    (600, 2560, 4096): (20.4, 16.9), (600, 4096, 256): (9.4, 8.4), (700, 2048, 512): (9.8, 8.4),
    (700, 10240, 256): (14.5, 15.8), (777, 14336, 512): (25.2, 22.6), (900, 64, 512): (6.7, 6.6),
    (900, 5120, 2048): (21.1, 18.4), (901, 5120, 2048): (21.1, 18.4), (901, 6144, 4096): (32.9, 28.8),
    (901, 10240, 8192): (70.3, 57.5), (1003, 96, 512): (7.6, 6.7), (1003, 1024, 14336): (48.0, 27.2),
    (1003, 2048, 1024): (12.6, 10.5), (1003, 6144, 1024): (17.6, 15.8), (1100, 4096, 4096): (32.8, 23.6),
    (1100, 28672, 512): (44.5, 41.0), (1280, 64, 768): (8.2, 7.0), (1280, 96, 1024): (10.2, 8.9),
    (1280, 1024, 256): (9.1, 7.6), (1280, 4096, 8192): (51.3, 39.9), (1280, 6144, 4096): (33.6, 35.4),
    (1500, 8, 4096): (21.8, 15.1), (1500, 64, 1024): (9.6, 8.9), (1500, 2048, 8192): (34.3, 30.0),
    (1650, 256, 4096): (21.6, 15.1), (1650, 256, 8192): (32.7, 20.3), (1650, 28672, 14336): (441.5, 414.2),
    (1800, 6144, 1024): (23.5, 21.5), (2000, 128, 1024): (11.8, 9.6), (2048, 8192, 8192): (93.5, 96.6),
    (2600, 6144, 8192): (102.1, 88.8), (2048, 6144, 4096): (46.8, 46.2),
    (2600, 2048, 2048): (23.0, 20.2), (2600, 2048, 14336): (92.4, 81.3), (3000, 256, 14336): (63.4, 44.1),
    (3000, 2048, 2048): (23.3, 21.0), (4096, 96, 1536): (15.1, 13.5), (5000, 2048, 1024): (25.0, 23.4),
    (6000, 28672, 512): (182.0, 194.7), (8192, 10240, 8192): (504.4, 470.4), (8192, 14336, 1024): (135.5, 145.4),
}
# us of SwiGLU blocks, tokens x d x d_ff, with packed and with one-byte codes in front of gate||up
MEASURED_BLOCKS = {
    (129, 256, 1024): (33.9, 17.5), (777, 4096, 14336): (182.7, 125.9), (1003, 4096, 14336): (181.0, 148.6),
    (1500, 2048, 5632): (90.9, 74.9), (3000, 4096, 11008): (303.6, 276.8), (4096, 512, 8192): (169.6, 184.1),
    (4096, 1024, 4096): (99.7, 107.8), (8192, 512, 2048): (91.4, 100.2), (8192, 1024, 4096): (183.3, 202.6),
    (8192, 8192, 28672): (3676, 3362),
}


def test_route_of_the_codes_is_the_faster_one_measured():
    """Either side of 900 tokens, few outputs, short rows, rounds of tiles that are filled and that are not."""
    for (M, N, K), us in MEASURED_SIDES.items():
        assert us[wt_ahead(M, N, K)] <= 1.06 * min(us), (M, N, K)
    for (M, d, d_ff), us in MEASURED_BLOCKS.items():
        assert us[wt_ahead(M, 2 * d_ff, d, swiglu=True)] <= 1.06 * min(us), (M, d, d_ff)
    assert not any(wt_ahead(M, N, K) for M in (1, 17, 64) for N in (8, 4096) for K in (128, 4096))
