"""The bf16 softmax head's tensor-core kernels at the edges of their tiles --
row groups of 16, blocks of 64 rows, features per lane, block and split, odd
widths -- held to the oracle as the head's own tests hold it; and the error of
their sums against 64 bits, which does not grow with the batch."""

import numpy as np
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


def _exact_features(torch, ff, layer, x):
    """The head's features (activity times row scale, one fp32 rounding each)
    of a one-layer net, read as logits through ten of them at a time."""
    n, F = x.shape[0], layer.out_features
    head = ff.Head(F, max_rows=n)
    A, z = torch.empty(n, F, device="cuda"), torch.empty(n, 10, device="cuda")
    for f in range(0, F, 10):
        k = min(10, F - f)
        V = np.zeros((10, F), np.float32)
        V[np.arange(k), f + np.arange(k)] = 1.0
        head.set_state(V=V, c=np.zeros(10, np.float32))
        head.predict([layer], x, logits=z)
        A[:, f:f + k] = z[:, :k]
    return A.double()


# Each term carries the roundings of dz (exp, sum, quotient, difference and the
# mean: 4), of its product with the row scale (1) and of its feature (1), and
# each 16-row sum is cut once (2): 8 x 2^-24 of the terms, whatever the batch.
# Left in the MMA accumulators the sum drifted by 1.5e-6 at 1024 rows and 1.9e-5
# at 16384.  Class 0 is nobody's label: all its terms have one sign.
@pytest.mark.parametrize("n", [1024, 16384])
def test_head_gradient_error_does_not_grow_with_the_batch(env, n):
    torch, ff = env
    F = 128
    g = torch.Generator("cuda").manual_seed(n)
    layer = ff.Layer(784, F, prec="bf16", init_seed=3)
    x = torch.rand(n, 784, device="cuda", generator=g)
    y = torch.randint(1, 10, (n,), device="cuda", dtype=torch.int32, generator=g)
    A = _exact_features(torch, ff, layer, x)
    head = ff.Head(F, max_rows=n)
    V = (np.random.default_rng(1).standard_normal((10, F)) * 0.3).astype(np.float32)
    head.set_state(V=V, c=np.zeros(10, np.float32))
    z = torch.empty(n, 10, device="cuda")
    head.predict([layer], x, logits=z)
    dz = (torch.softmax(z.double(), 1) - torch.nn.functional.one_hot(y.long(), 10).double()) / n
    head.train_step([layer], x, y)
    torch.cuda.synchronize()
    head.check()
    dV = torch.from_numpy(head.get_grad()[0]).cuda().double()
    bound = 8 * 2.0 ** -24
    ref, terms = dz.T @ A, dz.abs().T @ A
    assert bool(((dV - ref).abs() <= bound * terms).all()), float(((dV - ref).abs() / terms).max())
    assert float((dV[0] - ref[0]).norm() / ref[0].norm()) <= bound


# the feature's rounding, the cut of each 32-feature sum (2) and the rounded
# adds of 8 such sums, two halves, three parts and the splits, on random terms
@pytest.mark.parametrize("F", [256, 2000])
def test_head_logits_error(env, F):
    torch, ff = env
    n = 256
    layer = ff.Layer(784, F, prec="bf16", init_seed=3)
    x = torch.rand(n, 784, device="cuda", generator=torch.Generator("cuda").manual_seed(F))
    A = _exact_features(torch, ff, layer, x)
    head = ff.Head(F, max_rows=n)
    V = np.abs(np.random.default_rng(2).standard_normal((10, F))).astype(np.float32)
    head.set_state(V=V, c=np.zeros(10, np.float32))
    z = torch.empty(n, 10, device="cuda")
    head.predict([layer], x, logits=z)
    ref = A @ torch.from_numpy(V).cuda().double().T
    assert float((z.double() - ref).norm() / ref.norm()) <= 1.5 * 2.0 ** -24
