"""The fp32 GEMMs (CUDA cores, and bf16 parts on the tensor cores) at the edges
of their tiles, stages and K slices: forward and weight gradient of an fp32
layer against float64 products, within the bound of a K-term fp32 sum (K + 8
roundings of 2^-24 of the terms' absolute sum, whatever the order)."""

import numpy as np
import pytest

from oracle import ff_oracle as fo
from tests.gpu_common import U32, assert_adam_state, lib_ready, torch_cuda

pytestmark = pytest.mark.gpu

# rows 2B, K, N: one tile and less; tile edges +-1; widths off every
# multiple of 4 (unaligned weight rows); one and several K slices, ragged
# stages; outputs of many large tiles
SHAPES = [(2, 10, 8), (2, 33, 1), (62, 31, 63), (64, 32, 64), (66, 65, 65), (128, 784, 500), (130, 786, 129),
          (254, 1001, 127), (256, 256, 2000), (600, 129, 1023), (1538, 300, 1027),
          # large enough for the tensor cores: whole tiles; every edge ragged;
          # a last chunk of 4; several K slices, the last one short
          (512, 768, 2048), (1022, 1004, 1001), (1150, 2052, 643), (258, 2500, 1500),
          # forwards by CTA pairs: a last 256-column tile of 4 columns (its second half empty) and
          # a last row tile two rows short; two K slices
          (2046, 1004, 2052), (1022, 784, 2000)]


@pytest.mark.parametrize("M,K,N", SHAPES)
def test_fp32_forward_and_weight_gradient_at_tile_edges(M, K, N):
    torch = torch_cuda()
    ff = lib_ready()
    g = torch.Generator("cuda").manual_seed(M * 7 + K * 3 + N)
    layer = ff.Layer(K, N, prec="fp32", theta=2.0, lr=1e-3, keep_grad=True, max_rows=M)
    x = layer.new_activation(M, K)
    x[:, K:] = float("nan")  # the padding of an activation row is never read
    x[:, :K] = torch.rand(M, K, device="cuda", generator=g)
    s = (1.0 / torch.linalg.vector_norm(x[:, :K], dim=1)).contiguous()
    st = layer.get_state()
    b = (np.random.default_rng(1).standard_normal(N) * 0.05).astype(np.float32)
    layer.set_state(W=st["W"], b=b)
    W = torch.from_numpy(st["W"]).cuda().double()
    h = layer.new_activation(M)
    h.fill_(7.0)
    good = torch.empty(M, device="cuda")
    layer.train_step(x, row_scale=s, B=M // 2, h_out=h, goodness=good)
    torch.cuda.synchronize()
    layer.check()
    xs = x[:, :K].double() * s.double()[:, None]
    bd = torch.from_numpy(b).cuda().double()
    ref = torch.relu(xs @ W.T + bd)
    bound = (K + 8) * U32 * (xs.abs() @ W.abs().T + bd.abs())
    assert bool(((h[:, :N].double() - ref).abs() <= bound).all())
    assert bool((h[:, N:] == 0).all())
    gref = (ref * ref).sum(1)
    gb = (2 * ref * bound + bound ** 2).sum(1) + (N + 8) * U32 * gref
    assert bool(((good.double() - gref).abs() <= gb).all())
    # a layer that keeps no gradient ends in the same state (small shapes form
    # the gradient and the Adam step in one kernel)
    plain = ff.Layer(K, N, prec="fp32", theta=2.0, lr=1e-3, max_rows=M)
    plain.set_state(W=st["W"], b=b)
    plain.train_step(x, row_scale=s, B=M // 2)
    torch.cuda.synchronize()
    after, sp = layer.get_state(), plain.get_state()
    for k in ("W", "b", "mW", "vW", "mb", "vb"):
        assert np.array_equal(after[k], sp[k]), k
    # and W, m, v are Adam's on that gradient
    dw = layer.get_grad()[0].astype(np.float64)
    zero = np.zeros((N, K))
    assert_adam_state(after["W"], after["mW"], after["vW"], st["W"].astype(np.float64), zero, zero, 1, dw,
                      1e-6 * np.abs(dw) + 1e-12, fo.AdamHyper(lr=1e-3), "W")
    # the weight gradient of the GPU's own operand
    G = torch.from_numpy(layer.get_grad_operand(M)).cuda()[:, :N]
    dW = torch.from_numpy(layer.get_grad()[0]).cuda().double()
    xd = x[:, :K].double()
    assert bool(((dW - G.T @ xd).abs() <= (M + 8) * U32 * (G.abs().T @ xd.abs())).all())


# the first two take the tensor cores' bf16 parts, the last the CUDA cores
@pytest.mark.parametrize("M,K,N", [(512, 768, 2048), (2048, 2000, 2000), (64, 32, 64)])
def test_values_past_the_largest_bf16(M, K, N):
    """Finite values that bf16 rounds to infinity count like any other, and a
    sum that overflows to -inf is a zero activity, whatever the GEMM."""
    torch = torch_cuda()
    ff = lib_ready()
    g = torch.Generator("cuda").manual_seed(K)
    layer = ff.Layer(K, N, prec="fp32", max_rows=M)
    W = layer.get_state()["W"]
    W[0, 5], W[1, 5], W[2, 9] = 3.4e38, -3.4e38, -3e38
    layer.set_state(W=W, b=np.zeros(N, np.float32))
    x = layer.new_activation(M, K)
    x[:, :K] = torch.rand(M, K, device="cuda", generator=g)
    x[:, 5] = 2.0 ** -120   # times 3.4e38: 256
    x[:, 9] = 0.0
    x[7, 9] = 4.0           # row 7, unit 2: -1.2e39
    h = layer.new_activation(M)
    good = torch.empty(M, device="cuda")
    layer.forward(x, row_scale=torch.ones(M, device="cuda"), h_out=h, goodness=good)
    torch.cuda.synchronize()
    layer.check()           # nothing non-finite
    xd, Wd = x[:, :K].double(), torch.from_numpy(W).cuda().double()
    ref = torch.relu(xd @ Wd.T)
    bound = (K + 8) * U32 * (xd.abs() @ Wd.abs().T)
    assert bool(((h[:, :N].double() - ref).abs() <= bound).all())
    assert float(ref[0, 0]) > 100 and float(h[7, 2]) == 0.0


@pytest.mark.parametrize("M,K,N,kind", [(2048, 2000, 2000, "f32tc"), (128, 784, 500, "simt"), (2048, 2002, 2000, "mixed")])
def test_profile_names_the_kernels_that_ran(M, K, N, kind):
    import ctypes
    torch = torch_cuda()
    ff = lib_ready()
    layer = ff.Layer(K, N, prec="fp32", max_rows=M)
    x = layer.new_activation(M, K)
    x[:, :K] = 0.5
    s = torch.ones(M, device="cuda")
    lib = ff.lib()
    lib.ff_profile_enable(1)
    layer.train_step(x, row_scale=s, B=M // 2)
    torch.cuda.synchronize()
    lib.ff_profile_enable(0)
    names = (ctypes.c_char_p * 32)()
    n = lib.ff_profile_read(32, names, None, None, None)
    gemms = {names[i].decode() for i in range(n) if b"gemm" in names[i]}
    # K = 2002: the weights' rows are not 16-byte aligned, the activities' are
    assert gemms == {"f32tc": {"fwd_gemm_f32tc", "wgrad_gemm_f32tc"}, "simt": {"fwd_gemm_simt", "wgrad_gemm_simt"},
                     "mixed": {"fwd_gemm_simt", "wgrad_gemm_f32tc"}}[kind]
