"""A batch of one length class picks the score pass's rows per lane by its
number of pairs: batches on the way from the fewest rows to those of a full GPU,
bit-exact against the oracle."""
import numpy as np
import pytest

import synth
from gpu_helpers import assert_parity, run_gpu

pytestmark = pytest.mark.gpu

DEFAULT = (5, -4, -10, -1)


@pytest.mark.parametrize("n_pairs,m", [(4200, 100), (9000, 100), (16_384, 100), (40_000, 100), (16_384, 150),
                                       (16_384, 250), (5000, 500)])
def test_one_class(n_pairs, m):
    wl = synth.random_pairs(n_pairs, (m - 4, m), (m + 60, m + 100), seed=n_pairs + m, alphabet=3)
    got = run_gpu(wl, DEFAULT)
    pick = np.sort(np.random.default_rng(4).choice(n_pairs, 200, replace=False))
    assert_parity(wl, got, DEFAULT, pairs=pick)
