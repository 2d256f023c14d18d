"""The flop count of the warp-per-subaperture FP32 kernel that the bench's roofline divides, by hand from
the kernel's stages: an even compiled geometry, an odd one, and one of four-fold N that is not compiled
in (its columns do not fold twice)."""
import bench


def test_row_flops_by_hand():
    u = 4 * 32 * 5 * 10 + 4 * 32 * 10 + 4 * 32 * 5      # half sums, one exchange, the fold of the rows
    y = 32 * 16 * (5 * 8 + 4 + 2 * 3)                   # per lane 16 column pairs
    t = 32 * 8 * (8 + 5 * 8) + 16 * 10 * 4              # two column pairs and five column pairs of T; the fold
    am = 10 * 10 * (16 * 8 + 4 + 2 * 6 + 4)             # A of +-dy over 16 row pairs, K~ A twice, the fold
    q = 8 * 10 * (10 * 8 + 4)                           # row pairs x dx
    b = 16 * 8 * (5 * 8 + 4)                            # rows x column pairs
    assert bench.spot_flops(10, 32, 16, True, "spot_row_fp32_N32") == u + y + t + am + q + b + 6 * 256 == 75536
    assert bench.spot_flops(10, 32, 16, False, "spot_row_fp32_N32") == u + y + 32 * 32 + 6 * 256 == 36480
    u = 4 * 21 * 5 * 9 + 4 * 21 * 9 + 4 * 21 * 5
    y = 21 * 11 * (5 * 8 + 4 + 2 * 3)
    t = 21 * 11 * (2 + 9 * 4) + 11 * 9 * 4
    rest = 81 * (11 * 8 + 4 + 2 * 6 + 4) + 4 * 9 * (9 * 8 + 4) + 7 * 4 * (9 * 4 + 4) + 6 * 49
    assert bench.row_flops(9, 21, 7, True) == u + y + t + rest == 38578
    assert bench.row_flops(9, 21, 7, False) == u + y + 21 * 21 + 6 * 49 == 17241
    per_pair = bench.row_flops(7, 28, 14, True) - (4 * 28 * 4 * 7 + 4 * 28 * 7 + 4 * 28 * 4 + 28 * 14 * (8 * 4 + 10)
               + 4 * 14 * 7 + 49 * (8 * 14 + 20) + 7 * 7 * 60 + 14 * 7 * 32 + 6 * 196)
    assert per_pair == 28 * 14 * (2 + 4 * 7)
