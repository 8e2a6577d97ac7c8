"""The vocabulary pass at the edges of its chunking: one logit short of and beyond a batch of 4096, rows on and off 16-byte
boundaries, chunk counts around what the merge keeps in registers, maxima in the first and last logit and repeated across
batches, warps and chunks.  Against the oracle."""
import numpy as np
import pytest

from helpers import Dev
from test_gpu_scores_threshold import _compare_scored
from workloads import make_logits, make_mask

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return Dev()


def _inputs(B, L, V, seed):
    z = make_logits(B, L, V, (0.5, 6.0), seed)
    top = float(z.max()) + 1.0
    z[0, 0, 0] = top                                   # first logit
    z[0, 1, V - 1] = top                               # last logit
    z[0, 2, [V // 2, V - 1]] = top                     # twice: the lower index wins
    z[0, 3, V - 1] = z[0, 3, max(V - 4097, 0)] = top   # twice, a batch apart
    z[0, 4, : max(V - 2, 1)] = -float("inf")           # nothing finite but the end (V >= 3)
    return z


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("B,L,V", [(1, 33, 4095), (2, 17, 4096), (1, 9, 8193), (1, 32, 98304), (1, 8, 98304), (1, 8, 98305), (1, 8, 102401), (3, 40, 12288), (40, 32, 20484)])
def test_chunk_edges(dev, oracle, B, L, V, kind):
    masked0 = make_mask(B, L, L - 2, V).numpy()
    masked0[0, :5] = 1
    assert _compare_scored(dev, oracle, _inputs(B, L, V, B + L + V), masked0, 0, kind)


@pytest.mark.parametrize("L", [31, 32, 33, 64, 1024])
def test_ranking_of_short_and_long_blocks(dev, oracle, L):
    """Blocks whose rows are merged by eight lanes each (up to 32 positions) and by four, all ranked by eight lanes a position; k beyond and
    below the number of masked positions."""
    for k, n_masked in ((1, L), (7, L - 1), (L + 3, L // 2)) if L <= 64 else ((1, L), (L + 3, L // 2)):
        for seed in range(12):
            if _compare_scored(dev, oracle, make_logits(2, L, 513, (0.5, 6.0), 10 * L + seed), make_mask(2, L, n_masked, seed).numpy(), k, 0):
                break
        else:
            pytest.skip("near ties in every draw")


@pytest.mark.parametrize("L", [1, 32, 33, 100])
def test_tickets_of_few_masked_rows(dev, oracle, L):
    """Which blocks take a ticket: elements with no masked row, the first only, the last only, all but the first; twice, since
    the last block resets the count."""
    masked0 = np.zeros((4, L), np.uint8)
    masked0[1, 0] = masked0[2, L - 1] = masked0[3, 1:] = 1
    for _ in range(2):
        for k in (0, 1, 3):
            assert any(_compare_scored(dev, oracle, make_logits(4, L, 9001, (0.5, 6.0), 50 * L + seed), masked0, k, 0) for seed in range(12))


# more than 32 positions are merged by four lanes a row, which hold 20 chunks: exactly that many, one more, and more than a pass of 64 rows
@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("L,V", [(40, 163840), (40, 163841), (65, 98304), (130, 9000)])
def test_merge_of_long_blocks(dev, oracle, L, V, kind):
    masked0 = make_mask(1, L, L - 3, V).numpy()
    masked0[0, :5] = 1
    # (ranked: plain rows, since those of _inputs share their top logit, so that their scores are near ties in every draw)
    assert _compare_scored(dev, oracle, _inputs(1, L, V, L + V), masked0, 0, kind)
    for k in (3, L + 3):
        assert any(_compare_scored(dev, oracle, make_logits(1, L, V, (0.5, 6.0), L + V + seed), masked0, k, kind) for seed in range(12))


# rows of the same logits, hence the same score to the bit: the earlier position goes first, also when the two are eight positions or more
# apart (another lane's or another round's) and in different words of the set of chosen ones
@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("L,pair", [(32, (3, 11)), (32, (0, 31)), (40, (7, 39)), (130, (31, 32)), (130, (2, 129)), (1024, (100, 900))])
def test_identical_rows_far_apart(dev, oracle, L, pair, kind):
    z = make_logits(1, L, 513, (0.5, 2.0), L)
    z[0, pair[0]] = make_logits(1, 1, 513, (1.0, 1.0), 1)[0, 0]
    z[0, pair[0], 77] = 12.0                                      # 0.99 of the probability: the best row by every score
    z[0, pair[1]] = z[0, pair[0]]
    masked0 = np.ones((1, L), np.uint8)
    assert _compare_scored(dev, oracle, z, masked0, 1, kind) and _compare_scored(dev, oracle, z, masked0, 2, kind)
