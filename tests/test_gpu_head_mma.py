"""The bf16 softmax head's tensor-core kernels at the edges of their tiles --
row groups of 16, slabs of 512 rows, features per lane, block and split, odd
widths -- held to the oracle as the head's own tests hold it."""

import pytest

from tests.gpu_common import lib_ready, torch_cuda
from tests.test_gpu_head import test_head_predict_matches_oracle as predict_check
from tests.test_gpu_head import test_head_train_step_matches_oracle as step_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    return torch, lib_ready()


# one segment narrower than a block; one wider than a split by a few features;
# several segments that start off every multiple of 4 and 8
@pytest.mark.parametrize("dims,n", [((784, 31), 17), ((784, 523), 65), ((784, 64, 33, 131), 513),
                                    ((784, 72, 265, 257), 1024)])
def test_head_step_at_tile_edges(env, dims, n):
    step_check(env, "bf16", dims, n)


@pytest.mark.parametrize("dims,n,max_rows", [((784, 31), 1, 0), ((784, 64, 33, 1029), 79, 64)])
def test_head_predict_at_tile_edges(env, dims, n, max_rows):
    predict_check(env, "bf16", dims, n, max_rows)
