"""CPU: the form each launch takes, against both sides as measured on GB300 (the
times beside the cases): a form is not taken where the other one is faster."""
import pytest

import plan_host as P


@pytest.mark.parametrize("nx,ny,G,T,strips", [
    (1, 2_494_174, 608, 256, False),    # 7.4 us point by point, 138 in strips
    (2, 949_144, 608, 256, False),      # 7.1, 55.8
    (6, 362_425, 2389, 256, False),     # 9.0, 25.0
    (11, 131_295, 608, 256, False),     # 6.1, 10.3
    (21, 20_920, 608, 256, False),      # 3.2, 4.4
    (287, 710, 62, 1024, False),        # 3.1, 4.1
    (2061, 22, 176, 128, False),        # 2.0, 2.3
    (301, 300, 608, 256, False),        # 2.0, 2.5
    (30, 3078, 52, 128, True),          # 4.1, 3.2
    (33, 56_391, 608, 256, True),       # 7.2, 6.1
    (57, 89_460, 313, 32, True),        # 182, 72.6
    (217, 5887, 1158, 512, True),       # 6.8, 4.5
    (6193, 82, 608, 256, True),         # 3.3, 2.7
    (3001, 2503, 608, 256, True),       # 24.8, 13.8
    (4095, 4095, 608, 256, True),       # 54.7, 28.7
    (3, 2 ** 31, 608, 256, False),      # rows beyond 32 bits
])
def test_auto_stencil2d_strips(nx, ny, G, T, strips):
    assert P.cols(nx, ny, G, T) == strips


@pytest.mark.parametrize("body,n,sched,chunk,G,T", [
    ("axpy", 2_050_019, P.CHUNKED, 64, 3, 64),       # 261 us staged, 402 in rows, 394 plain
    ("axpy", 135_387, P.DYNAMIC, 64, 1, 64),         # 65, 59, 99
    ("axpy", 20_319, P.NONMONO, 256, 2, 32),         # 12, 16, 16
    ("load_i64", 256_999, P.DYNAMIC, 32, 4, 64),     # 52, 63, 63
    ("axpy", 300_007, P.DYNAMIC, 64, 1, 32),
    ("load_i32", 300_007, P.CHUNKED, 64, 8, 64),     # 7 blocks of 37,501, one of 37,500
    ("axpy", 1 << 26, P.DYNAMIC, 256, 4096, 32),
])
def test_staged_where_every_block_starts_on_16_bytes(body, n, sched, chunk, G, T):
    q, r = divmod(n, G)
    aligned = all((g * q + min(g, r)) * P.BODIES[body][1] % 16 == 0 for g in range(G))
    assert (P.stream(body, n, sched, chunk, G, T)[0] == "staged") == aligned
    assert P.stream(body, n, sched, chunk, G, T, stage_bytes=0)[0] == "plain"
    assert P.stream(body, n + 16 * G, sched, chunk, G, T)[0] == \
        P.stream(body, n, sched, chunk, G, T)[0]


@pytest.mark.parametrize("body,elem", [("axpy", 4), ("load_i64", 8)])
def test_blocks_aligned_is_exact(body, elem):
    """The rule for blocks that start on 16 bytes against every block's start."""
    for G in (1, 2, 3, 4, 5, 7, 8, 12):
        for n in range(G * 2560, G * 2563):
            q, r = divmod(n, G)
            aligned = all((g * q + min(g, r)) * elem % 16 == 0 for g in range(G))
            assert (P.stream(body, n, P.DYNAMIC, 256 // elem, G, 32)[0] == "staged") == aligned, \
                (G, n)


@pytest.mark.parametrize("body,n,sched,chunk,G,T,rows", [  # plain and rows in us
    ("load_i64", 1_411_583, P.CHUNKED, 50, 6, 32, False),       # 180, 396
    ("load_bf16_sum", 5_276_959, P.STATIC, 0, 9, 32, False),    # 136, 262
    ("load_f32_max", 6_639_461, P.CHUNKED, 4096, 23, 32, False),  # 112, 176
    ("load_i32", 12_784_957, P.DYNAMIC, 40, 608, 256, False),   # 20.3, 30.5
    ("load_i64", 428_377, P.DYNAMIC, 50, 1, 32, False),         # 452, 710
    ("load_bf16_sum", 9_407_331, P.DYNAMIC, 100, 35, 1024, False),  # 26.6, 38.2
    ("dot", 785_073, P.CHUNKED, 40, 2, 64, False),              # 242, 402
    ("axpy_sum", 147_889, P.GUIDED, 256, 2, 32, False),         # 92, 136
    ("axpy", 5_143_369, P.CHUNKED, 50, 608, 256, False),        # 15.4, 23.9
    ("axpy", 3_030_322, P.CHUNKED, 40, 9, 32, False),           # 630, 789
    ("axpy_i32_sum", 11_984_041, P.STATIC, 0, 608, 256, False),  # 37.1, 43.3
    ("axpy", 67_108_864, P.DYNAMIC, 256, 608, 256, True),       # 197, 135
    ("axpy", 50_000_001, P.STATIC, 0, 1184, 256, True),         # 124, 102
    ("axpy_i32_sum", 1 << 20, P.STATIC, 0, 4, 128, True),       # 59.8, 53.7
    ("axpy", 1_447_680, P.GUIDED, 64, 39, 256, True),           # 69.3, 14.6
    ("axpy", 45_266_466, P.CHUNKED, 50, 231, 64, True),         # 356, 222
    ("dot", 30_055_685, P.DYNAMIC, 128, 18, 512, True),         # 491, 232
    ("load_f32_max", 62_239_855, P.DYNAMIC, 128, 3, 1024, True),  # 3044, 1398
    ("load_i32", 18_047_637, P.DYNAMIC, 4096, 26, 512, True),   # 140, 73
    ("load_f32_max", 58_005_398, P.STATIC, 0, 153, 64, True),   # 138, 79
])
def test_rows_where_they_gain(body, n, sched, chunk, G, T, rows):
    assert (P.stream(body, n, sched, chunk, G, T)[0] == "rows") == rows


@pytest.mark.parametrize("n,sched,chunk,G,T,pieces", [  # plain and pieces in us
    (1_515_221, P.CHUNKED, 40, 6, 64, False),       # 173, 440
    (2_356_909, P.STATIC, 0, 26, 32, False),        # 58, 120
    (902_283, P.CHUNKED, 1000, 3, 32, False),       # 220, 427
    (239_777, P.DYNAMIC, 40, 1, 64, False),         # 144, 315
    (1_778_248, P.DYNAMIC, 500, 18, 32, False),     # 81, 167
    (1_382_429, P.NONMONO, 256, 164, 512, False),   # 12.3, 18.8
    (5_700_616, P.DYNAMIC, 256, 608, 256, False),   # 17.1, 21.3
    (3_459_739, P.DYNAMIC, 50, 426, 1024, False),   # 16.6, 23.1
    (1 << 26, P.CHUNKED, 64, 608, 256, True),       # 210, 129
    (1 << 26, P.DYNAMIC, 256, 608, 256, True),      # 151, 143
    (1 << 24, P.CHUNKED, 32, 608, 256, True),       # 78, 42
    (1 << 24, P.DYNAMIC, 64, 608, 256, True),       # 58, 36
    (66_684_445, P.NONMONO, 50, 662, 256, True),    # 258, 162
    (16_870_783, P.DYNAMIC, 40, 133, 32, False),    # 237, 299
    (502_472, P.DYNAMIC, 100, 30, 1024, False),     # 7.7, 9.3
    (134_259, P.CHUNKED, 500, 1, 256, False),       # 37.4, 42.3
    (72_320, P.STATIC, 0, 4, 256, False),           # 6.4, 7.3
    (1_936_512, P.STATIC, 0, 79, 256, True),        # 11.9, 8.2
    (8_446_615, P.DYNAMIC, 64, 28, 128, True),      # 197, 158
    (2_005_184, P.DYNAMIC, 1000, 1, 512, True),     # 404, 292
    (62_584_413, P.DYNAMIC, 40, 608, 256, True),    # 180, 139
    (1_500_488, P.DYNAMIC, 50, 5, 1024, True),      # 95.8, 78.0
])
def test_stencil1d_pieces_where_they_gain(n, sched, chunk, G, T, pieces):
    assert P.line(n, sched, chunk, G, T) == pieces


@pytest.mark.parametrize("nseg,avg,G,T,dot,tiled", [  # plain and tiled in us
    (2226, 342, 161, 256, False, False),        # 31, 52
    (9044, 36, 524, 256, True, False),          # 42, 133
    (13_158, 150, 2704, 256, True, False),      # 58, 184
    (182, 450, 2731, 256, False, False),        # 6.1, 24.2
    (12_501, 5342, 546, 256, False, False),     # 277, 488
    (6879, 94, 3005, 32, True, False),          # 11.6, 29.5
    (9367, 66, 1251, 128, False, False),        # 34.8, 47.4
    (27, 58, 152, 256, True, False),            # 4.0, 4.4
    (4096, 13_280, 152, 256, False, True),      # 434, 199
    (963, 10_000, 18, 32, True, True),          # 2068, 292
    (568, 13_000, 1765, 32, False, True),       # 418, 101
    (2370, 3505, 960, 128, False, True),        # 47, 30
    (3906, 7800, 7, 128, False, True),          # 4199, 1407
    (97, 363, 1020, 32, True, True),            # 6.8, 5.3
    (132, 369, 906, 64, False, True),           # 8.5, 7.0
    (2001, 31, 1107, 32, True, False),          # 6.7, 10.9
])
def test_generic_tiles_where_they_gain(nseg, avg, G, T, dot, tiled):
    assert (P.tiles(nseg * avg, nseg, G, T, dot) > 0) == tiled


def test_generic_tile_rings_fit():
    """Rings of every team size lie beside the stack in the shared memory of one SM."""
    for T in range(32, 513, 32):
        for G in (1, 152, 153, 304, 305, 456, 608, 5000):
            for stack in (0, 4096, 48 * 1024, 150 * 1024, 226 * 1024):
                t = P.tiles(1 << 30, 64, G, T, stack=stack)
                assert t == 0 or 2 <= t <= 8 and T <= 480


@pytest.mark.parametrize("n,sched,G,T,plain", [  # without overlap and with, us
    (1291 * 634, P.CHUNKED, 842, 128, True),        # 7.1, 8.6
    (33 * 782 * 128, P.STATIC, 782, 128, True),     # 51, 64
    (59 * 345 * 256, P.CHUNKED, 345, 256, True),    # 24, 29
    (1960 * 21, P.STATIC, 161, 256, False),         # 2.3, 1.9
    (3 * 4534, P.STATIC, 629, 32, False),           # 2.3, 1.8
    (461 * 145, P.DIST, 577, 256, False),           # 3.2, 2.6
    (1024 * 1024, P.CHUNKED, 2048, 32, False),      # 6.4, 5.8
    (1024 * 1024, P.STATIC, 2048, 32, False),       # 6.2, 5.8
    (22 * 12_345, P.DIST, 202, 64, False),          # 8.9, 8.3
    (7 * 33_202, P.STATIC, 205, 128, False),        # 3.5, 3.3
    (1 << 24, P.STATIC, 100, 256, False),           # less than a block an SM
])
def test_stencil2d_launch_overlap(n, sched, G, T, plain):
    assert P.uneven(n, sched, G, T) == plain


@pytest.mark.parametrize("nx,ny,sched,chunk,G,T,window", [  # the others and windows in us
    (4096, 4096, P.CHUNKED, 8, 8192, 32, False),       # 36, 88
    (4096, 4096, P.CHUNKED, 8, 1024, 32, False),       # 90, 176
    (2048, 2048, P.STATIC, 0, 4096, 64, False),        # 12, 20
    (4096, 4096, P.DYNAMIC, 100, 8192, 32, False),     # 45, 74
    (4096, 4096, P.DYNAMIC, 256, 8192, 32, False),     # 53, 96
    (4096, 4096, P.DYNAMIC, 256, 16_000, 32, False),   # 105, 158
    (4096, 4096, P.DYNAMIC, 100, 2048, 32, False),     # 41, 74
    (4096, 4096, P.NONMONO, 100, 16_000, 32, False),   # 81, 111
    (16, 306_391, P.DYNAMIC, 1000, 1091, 64, False),   # 52, 99
    (2048, 39, P.DYNAMIC, 1000, 39, 32, False),        # 14, 27
    (5, 1737, P.DYNAMIC, 32, 3378, 256, False),        # 13.7, 21.4
    (3, 444_749, P.CHUNKED, 8, 864, 1024, False),      # 17.0, 24.1
    (4096, 47, P.CHUNKED, 16, 188, 1024, False),       # 6.5, 9.0
    (4096, 4096, P.CHUNKED, 64, 608, 256, True),       # 65, 52
    (4096, 4096, P.STATIC, 0, 608, 256, True),         # 59, 38
    (4096, 4096, P.DYNAMIC, 256, 608, 256, True),      # 64, 49
    (3001, 2503, P.CHUNKED, 61, 608, 256, True),       # 37, 24
    (4096, 4096, P.CHUNKED, 64, 16_000, 32, True),     # 252, 96
    (7343, 40, P.CHUNKED, 500, 738, 1024, True),       # 382, 67
    (6054, 913, P.CHUNKED, 16, 565, 1024, True),       # 71, 37
    (8, 1_741_190, P.CHUNKED, 16, 9519, 32, True),     # 148, 53
    (2548, 5652, P.CHUNKED, 32, 276, 32, False),       # 147, 250
    (2393, 6233, P.CHUNKED, 32, 297, 64, False),       # 109, 146
    (5798, 2480, P.CHUNKED, 32, 596, 32, False),       # 102, 269
    (847, 6781, P.CHUNKED, 40, 181, 32, True),         # 149, 102
    (5536, 2774, P.CHUNKED, 32, 897, 32, True),        # 193, 119
    (192, 61_956, P.CHUNKED, 32, 265, 64, True),       # 327, 127
    (5088, 1655, P.CHUNKED, 61, 628, 32, True),        # 141, 71
    (4, 2_597_540, P.CHUNKED, 50, 220, 32, True),      # 7989, 205
    (174, 68_534, P.CHUNKED, 256, 219, 128, True),     # 69, 52
    (64, 672, P.CHUNKED, 8, 14, 64, True),             # 13.3, 7.6
    (25, 33_226, P.CHUNKED, 16, 608, 256, True),       # 10.8, 7.6
])
def test_stencil2d_windows_where_they_gain(nx, ny, sched, chunk, G, T, window):
    assert P.window(nx, ny, sched, chunk, G, T) == window
    assert not P.window(nx, ny, sched, chunk, G, T, budget=16)
