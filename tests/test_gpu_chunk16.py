"""The 16-token chunk engine (split-fp16 tensor-core products at fp32 precision) at the sizes where it can go wrong:
lengths around a chunk and around the ring of four operand tiles, every block of value columns, both key sizes, and
decays too strong to be divided by inside a chunk."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from tests.test_gpu_parity import all_pairs, check_backward, check_forward, upstream

# Operands keep 22 bits and the products of their tails (2^-22) are left out; sums are fp32 over at most 128 terms,
# carried over chunks by a contraction.  That is a few 1e-7 of a tensor's largest entry (8e-7 measured); ten times that.
TOL = 1e-5


@pytest.mark.parametrize("B,H,T,d_k,d_v,alpha", [
    (1, 2, 1, 128, 128, "u(0.9,1)"), (1, 2, 15, 64, 64, "u(0.9,1)"), (2, 1, 16, 128, 64, "u(0.9,1)"),
    (1, 3, 17, 64, 128, "u(0.9,1)"), (1, 2, 65, 128, 128, "u(0.3,1)"), (1, 1, 333, 128, 128, "sigmoid(n(3,1))"),
    (3, 16, 37, 128, 128, "u(0.9,1)"), (5, 16, 33, 128, 128, "u(0.9,1)"), (5, 16, 81, 64, 128, "u(0.9,1)"),
    (1, 2, 200, 128, 128, "u(0.0,1)"), (5, 16, 40, 64, 64, "u(0.0,0.02)")])
def test_fp32_forward(B, H, T, d_k, d_v, alpha):
    cfg = workloads.CONFIGS[0].scaled(name="c16", B=B, T=T, H=H, d_k=d_k, d_v=d_v, chunk=64, alpha=alpha, s0_std=0.5,
                                      seed=300 + T + H)
    inp = workloads.forward_inputs(cfg)
    if alpha.startswith("u(0.0"):
        inp["alpha"][:, ::17, :, ::5] = 0.0
    inp["v"] *= np.exp2(np.arange(d_v) % 24 - 12).astype(np.float32)      # value channels of very different size
    check_forward(cfg, inp, all_pairs(cfg)[:6] + all_pairs(cfg)[-2:], TOL)


# The gradients chain four such products and a sum over up to 64 tokens (D): five times the forward's bound.
BWD_TOL = 5e-5


@pytest.mark.parametrize("B,H,T,d_k,d_v,alpha,im", [
    (1, 2, 15, 128, 128, "u(0.9,1)", True), (1, 2, 16, 64, 64, "u(0.9,1)", False), (2, 1, 17, 128, 64, "u(0.9,1)", True),
    (1, 3, 64, 64, 128, "u(0.9,1)", False), (1, 2, 65, 128, 128, "u(0.3,1)", True), (1, 1, 225, 128, 128, "sigmoid(n(3,1))", False),
    (3, 16, 81, 128, 128, "u(0.9,1)", True), (5, 16, 97, 128, 128, "u(0.9,1)", False), (5, 16, 130, 64, 128, "u(0.9,1)", True),
    (5, 16, 70, 64, 64, "u(0.0,1)", True), (5, 16, 70, 128, 128, "u(0.0,0.1)", True), (1, 2, 80, 128, 128, "u(0.0,0.02)", False)])
def test_fp32_backward(B, H, T, d_k, d_v, alpha, im):
    cfg = workloads.CONFIGS[0].scaled(name="c16b", B=B, T=T, H=H, d_k=d_k, d_v=d_v, chunk=64, alpha=alpha, s0_std=0.5,
                                      seed=400 + T + H)
    inp = workloads.forward_inputs(cfg)
    if alpha.startswith("u(0.0"):
        inp["alpha"][:, ::17, :, ::5] = 0.0
    check_backward(cfg, inp, upstream(cfg, T, want_im=im), all_pairs(cfg)[:4] + all_pairs(cfg)[-2:], BWD_TOL)


@pytest.mark.parametrize("B,H,T,d_k,d_v,im", [
    (1, 149, 300, 128, 128, True), (5, 37, 200, 128, 64, False), (2, 100, 64, 64, 128, True), (1, 256, 130, 128, 128, False),
    (3, 99, 449, 64, 64, True)])
def test_backward_of_pairs_shared_by_two_blocks(B, H, T, d_k, d_v, im):
    """More pairs than SMs: nearly every pair is begun by one block and finished by the next, from a different place on."""
    cfg = workloads.CONFIGS[0].scaled(name="c16s", B=B, T=T, H=H, d_k=d_k, d_v=d_v, chunk=64, alpha="u(0.9,1)", s0_std=0.5,
                                      seed=500 + T + H)
    pairs = all_pairs(cfg)
    check_backward(cfg, workloads.forward_inputs(cfg), upstream(cfg, T, want_im=im), pairs[::19] + pairs[-2:], BWD_TOL)
