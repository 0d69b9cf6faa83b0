"""Both tile widths of the GEMM at the line between them (one round of narrow tiles over 74 CTA pairs) and where the
narrow one's operand ring wraps: exact cases, bit for bit against the oracle."""
import numpy as np
import pytest

from oracle import pq_oracle as O
from test_gpu_gemm import bf16_round, gemm, pack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(300, 4736, 128), (300, 4744, 128),            # 74 narrow tiles; 76: the wide one
                                   (256, 128, 64), (1, 8, 2048), (257, 136, 2112),  # 1, 8 and 9 K steps, ragged edges
                                   (130, 264, 4352)])                             # the ring wraps twice
def test_exact_at_the_line(M, N, K):
    rng = np.random.default_rng(M + N + K)
    pick = np.array([0, 2, 4, 10, 12], np.uint8)
    xn, wn = pick[rng.integers(0, 5, (M, K))], pick[rng.integers(0, 5, (N, K))]
    pow2 = np.array([0x30, 0x38, 0x40, 0x48], np.uint8)             # 0.5, 1, 2, 4
    sfx, sfw = pow2[rng.integers(0, 4, (M, K // 16))], pow2[rng.integers(0, 4, (N, K // 16))]
    Y = gemm(pack(xn), sfx, 0.5, pack(wn), sfw, 4.0, ldy=N + 8)
    assert np.array_equal(Y, bf16_round(O.gemm_ref(pack(xn), sfx, 0.5, pack(wn), sfw, 4.0)))


@pytest.mark.parametrize("M,N,K", [(2, 4736, 128), (2, 4744, 320), (3, 4744, 128), (1, 9472, 192), (16, 4744, 3136), (17, 4744, 3136),    # 37 and 38 narrow tiles, few rows
                                   (8, 4864, 1280), (8, 4872, 1280), (7, 4744, 1088), (16, 6272, 768), (3, 6280, 768)])    # 38 and 39; 49 and 50
def test_few_rows_at_the_line(M, N, K):
    test_exact_at_the_line(M, N, K)


# Two and three rounds of wide tiles; 1, 2, 3 and 4 blocks of 64 channels in the last K step; six K steps, so that the ring of five stages
# (and the scale slots) wraps inside a tile; a last row block of either operand that is the second of its tile or past the end.
@pytest.mark.parametrize("M,N,K", [(2200, 2440, 64), (4700, 1288, 384), (1025, 8200, 704), (2200, 2440, 512), (1100, 4744, 1472)])
def test_rounds_at_ragged_edges(M, N, K):
    test_exact_at_the_line(M, N, K)
