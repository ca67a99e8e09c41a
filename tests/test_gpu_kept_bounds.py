"""Upper bounds of what the first cut keeps, from the tokens near the query first: documents with more near tokens than are
collected at a time, masks whose last word is partial, every row width, and both sides of the rule that skips the step."""
import numpy as np
import pytest

from test_gpu_batch_scan import check, corpus, queries

pytestmark = pytest.mark.gpu


# D, q_len, centroids, documents, shortest, longest, queries, nprobe, n_prune
@pytest.mark.parametrize("call", [
    (32, 32, 1_029, 9_000, 1, 400, 257, 4, 260),         # 32-byte rows
    (32, 64, 2_047, 3_000, 500, 1_500, 220, 1, 300),     # 64-byte rows, hundreds of near tokens
    (64, 90, 999, 3_000, 300, 900, 220, 1, 300),         # 128-byte rows
    (64, 50, 1_500, 6_000, 100, 500, 165, 1, 400),       # ... of other query lengths
    (32, 100, 1_000, 9_000, 20, 90, 330, 2, 200),        # too many near tokens: all rows at once
    (32, 32, 1_029, 9_000, 1, 400, 41, 4, 60),           # too few documents: the same
    (128, 32, 120_003, 20_000, 90, 160, 250, 32, 263),   # 6-bit codes
    (32, 40, 107_001, 9_000, 150, 250, 220, 16, 300),    # ... without a mask
])
def test_kept_candidates_are_bounded_like_the_oracle_orders_them(call):
    arrays = corpus(*call)
    check(arrays, queries(np.random.default_rng(call[1]), arrays[0], call[6], call[1]), call[7], call[8])
