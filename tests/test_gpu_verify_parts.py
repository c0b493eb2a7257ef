"""The verification kernel splits a request's vocabulary over 8, 4, 2 or 1 CTAs (by the number of requests and of 4096-token
chunks): every split, with vocabularies that end in the middle of a part, leave parts empty, or fill them, against the oracle
as in test_gpu_verify."""
import numpy as np
import pytest

from paper_2410_11744_b200 import workloads as wl
from test_gpu_verify import B, check   # noqa: F401  (B is the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_req", [1, 18, 19, 37, 38, 74, 75])
@pytest.mark.parametrize("vocab", [4096, 4100, 8196, 12300, 16384, 20484, 32000, 32768])
def test_every_split_of_the_vocabulary(B, vocab, n_req):  # noqa: F811
    rng = np.random.default_rng(vocab + n_req)
    # chains accept and move on, stars reject one branch after the other
    trees = [wl.chain_tree(4) if r % 3 == 0 else np.concatenate([[-1], np.zeros(4, np.int32)]).astype(np.int32) if r % 3 == 1
             else wl.greedy_tree(rng, 6, 3, 0.5) for r in range(n_req)]
    case = wl.make_verify_case(vocab + n_req, vocab, trees, sharpness=2.0, disagreement=(0.2, 1.5)[n_req & 1])
    check(B, case, bonus=bool(vocab & 4), max_excused=1 + n_req // 25)


@pytest.mark.parametrize("n_req", [1, 18, 37, 74])
@pytest.mark.parametrize("bonus", [True, False])
def test_requests_that_reach_an_exchange_at_once(B, n_req, bonus):  # noqa: F811
    """Single nodes (with the bonus token: a draw straight away; without: no exchange at all), pairs and empty requests beside
    each other: the shortest way from a CTA's start to its first store into another's memory, and the ways around it."""
    trees = [wl.chain_tree(1 + r % 2) if r % 5 else np.zeros(0, np.int32) for r in range(1, n_req + 1)]
    case = wl.make_verify_case(n_req, 32000, trees, sharpness=2.0, disagreement=1.5)
    for _ in range(3):
        check(B, case, bonus=bonus, max_excused=1 + n_req // 25)
