"""Commit behind the acceptance of the same call: a thread's first request and first page slot are gone through before the
acceptance counts are there, the others behind.  On both sides of one request a thread; the largest batch has more page slots than threads."""
import numpy as np
import pytest

from gpu_util import REL_LARGE, run_and_check_pass
from lr_workloads import Model
from lr_workloads.gen import _finish
from paper_2506_19830_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_req,most", [(1, 20), (255, 40), (256, 40), (257, 40), (520, 600)])
def test_pass(n_req, most):
    rng = np.random.Generator(np.random.PCG64(n_req))
    reqs = []
    for _ in range(n_req):
        segs = [int(x) for x in rng.integers(1, 20, size=int(rng.integers(0, 12)))]
        depths = sorted(int(x) for x in rng.integers(0, len(segs) + 1, size=int(rng.integers(1, 12))))
        reqs.append({"P": int(rng.integers(0, most)), "segs": segs, "branches": [(g, 3, 2, 3) for g in depths]})
    w = _finish("commit", 5, Model(2, 1, 64, 64), reqs, rng, 0.4, 0.8, True, True, "nan")
    run_and_check_pass(w, path=B.PATH_GENERIC, rel_large=REL_LARGE)
