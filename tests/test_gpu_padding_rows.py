"""Query tiles whose padding begins anywhere in a warp's 32 rows: on both sides of every warp boundary of one tile and of the
second, with another request's queries behind the padding."""
import numpy as np
import pytest

from gpu_util import REL_LARGE, run_and_check_pass
from lr_workloads import Model
from lr_workloads.gen import _finish
from paper_2506_19830_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("q_len", [1, 31, 32, 33, 64, 65, 96, 97, 127, 128, 129, 160, 161, 225])
def test_padding(q_len, head_dim):
    rng = np.random.Generator(np.random.PCG64(q_len))
    reqs = [{"P": 400 + q_len, "segs": [9], "branches": [(1, q_len, q_len, 1)]}, {"P": 130, "segs": [5], "branches": [(1, 140, 140, 2)]}]
    w = _finish("padding", 5, Model(2, 2, head_dim, 1000), reqs, rng, 0.5, 0.6, True, True, "nan")
    run_and_check_pass(w, path=B.PATH_TENSOR_CORE, rel_large=REL_LARGE)
