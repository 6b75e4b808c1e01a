"""Edges of the element-wise kernels' splits: the PO block gradient at widths
that are and are not whole octets, and predictions that span more than one
group of layer-1 chunks."""

import numpy as np
import pytest

from paper_2404_08573_gb300 import synth
from tests.gpu_common import assert_close, lib_ready, torch_cuda
from tests.test_gpu_po import test_po_step_matches_oracle as po_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    return torch, lib_ready()


# a partial last octet, a partial last block of 256 columns, one row past a block of 32
@pytest.mark.parametrize("prec,N,n", [("bf16", 131, 33), ("bf16", 264, 31), ("fp32", 260, 33), ("fp32", 257, 1)])
def test_po_step_at_width_edges(env, prec, N, n):
    po_check(env, prec, False, 72, N, n)


# 4096 units: a group holds about 5100 samples (96 MB of operand and base rows)
@pytest.mark.parametrize("prec", ["bf16", "fp32"])
def test_predict_over_two_groups(env, prec):
    torch, ff = env
    n, dims = 5200, (784, 4096, 64)
    layers = [ff.Layer(dims[i], dims[i + 1], prec=prec, init_seed=80 + i) for i in range(2)]
    x = torch.from_numpy(synth.mnist_like(n, seed=82)).cuda()
    G = torch.empty(n, 10, device="cuda")
    P = torch.empty(n, 10, device="cuda")
    pred, _ = ff.predict(layers, x, goodness=G)
    for i in range(0, n, 1300):  # one group each
        ff.predict(layers, x[i:i + 1300], goodness=P[i:i + 1300])
    torch.cuda.synchronize()
    layers[0].check()
    # bf16: the same activations, so only the order of 64 non-negative squares
    # differs (64 x 2^-23); fp32: also the order of layer 1's sums, each side
    # within the 1e-4 that predictions are held to against the oracle
    assert_close(G.cpu().numpy(), P.cpu().numpy(), 64 * 2.0 ** -23 if prec == "bf16" else 2e-4, 0, "goodness")
    assert np.array_equal(pred.cpu().numpy(), G.cpu().numpy().argmax(axis=1))


# 784-2000x4 in fp32: chunks of 460 samples fill the GPU and take three TF32
# products a term; the last 80 samples, and small calls, take exact products.
# Each form is within 1e-4 of the exact goodness (the bound that predictions
# are held to against the oracle), so two calls differ by 1e-4 of it (half each:
# the exact form errs by less than 1e-6); the exact forms among themselves by
# the order of their sums: (4 layers of 2000 terms, square) 2 x 4 x sqrt(2000) x
# 2^-24 = 2.1e-5 at the very most, 2e-6 on random signs.
def test_fp32_prediction_alone_in_a_full_chunk_and_in_a_tail(env):
    torch, ff = env
    n, dims = 1000, (784, 2000, 2000, 2000, 2000)
    layers = [ff.Layer(dims[i], dims[i + 1], prec="fp32", init_seed=60 + i) for i in range(4)]
    x = torch.from_numpy(synth.mnist_like(n, seed=61)).cuda()

    def goodness(rows):
        G = torch.empty(rows.shape[0], 10, device="cuda")
        pred, _ = ff.predict(layers, rows, goodness=G)
        torch.cuda.synchronize()
        assert np.array_equal(pred.cpu().numpy(), G.cpu().numpy().argmax(axis=1))
        return G.double()

    def apart(a, b):
        return float(((a - b).abs() / b).max())

    G = goodness(x)
    small = goodness(x[:80])
    assert apart(G[:80], small) <= 1e-4          # a full chunk against a small call
    assert apart(G[920:], goodness(x[920:])) <= 2e-6   # the tail against a call of its own
    one = torch.cat([goodness(x[i:i + 1]) for i in range(8)])
    assert apart(one, small[:8]) <= 2e-6         # single samples against a small call
    layers[0].check()
