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
