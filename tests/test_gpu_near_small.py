"""The stored split-BF16 near field of small batches on CUDA cores (tiles cut into parts, partial
sums added in order): theta -> 0 makes it the whole potential, held against the oracle's direct sum.
Coefficients carry 16 significant bits, M 24: ~1e-5 of the cancelling terms, as for the tensor-core
tiles, whose bar (test_gpu_near_tc) is the same."""
import numpy as np
import pytest
import torch

from paper_1606_00247_gb300 import inputs

pytestmark = pytest.mark.gpu


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# every slice width (1, 2, 4, 8, 16), ragged ones, several slices, the last batch of the rule and the
# first that goes to the tensor cores (a ball of one or two tiles takes three slices per wave and more)
@pytest.mark.parametrize("B", [1, 2, 3, 7, 8, 9, 16, 17, 33, 64, 65])
def test_small_batches_vs_direct_sum(orc, B):
    from paper_1606_00247_gb300.api import Plan

    nodes, tets = inputs.sphere(h=0.25)
    M = inputs.gaussian_unit_m(nodes.shape[0], batch=B, seed=600 + B)
    plan = Plan(nodes, tets, p=2, leaf_size=16, theta=1e-9, precision="bf16x3", near_mode=1, max_batch=B)
    assert plan.stats()["n_near_tiles"] > 0
    u, H = plan.eval(torch.as_tensor(M, device="cuda"))
    u2, H2 = plan.eval(torch.as_tensor(M, device="cuda"))
    assert torch.equal(u, u2) and torch.equal(H, H2)
    for k in sorted({0, B // 2, B - 1}):
        assert rel_l2(u[k].cpu().numpy(), orc.direct(nodes, tets, M[k])) < 3e-5


# Saturated and slowly varying states: the 16 bits of W act on M - Mbar (Mbar: a mean over the tile),
# S_i . Mbar is FP32.  Uniform M leaves S_i . Mbar alone: S, Mbar, three products, their sum and u rounded
# to 2^-24 each, at most 7 * 2^-25 = 2e-7 of the largest term on average; 1 % of noise adds 1 % of the
# 2.4e-6 of a random M, the slow change 5e-8 (seen).  H differentiates the rounding of u: twice that.
# (The 16 bits of W on the full M: 4.8e-7 and 1.1e-6.)
@pytest.mark.parametrize("B", [1, 4, 8, 17, 64])
@pytest.mark.parametrize("kind", ["uniform", "noise", "slow"])
def test_nearly_uniform_states(orc, kind, B):
    from paper_1606_00247_gb300.api import Plan

    nodes, tets = inputs.sphere(h=0.25)
    r = np.random.default_rng(40 + B)
    M = np.tile(r.standard_normal((B, 1, 3)), (1, nodes.shape[0], 1))
    M /= np.linalg.norm(M, axis=2, keepdims=True)
    if kind == "noise":
        M += 0.01 * r.standard_normal(M.shape)
    if kind == "slow":
        M += 0.1 * np.sin(nodes @ r.standard_normal((3, 3)))
    M /= np.linalg.norm(M, axis=2, keepdims=True)
    u, H = Plan(nodes, tets, p=2, leaf_size=16, theta=1e-9, precision="bf16x3", near_mode=1, max_batch=B).eval(
        torch.as_tensor(M, device="cuda"))
    for k in sorted({0, B - 1}):
        ref = orc.direct(nodes, tets, M[k])
        assert rel_l2(u[k].cpu().numpy(), ref) < 2e-7
        assert rel_l2(H[k].cpu().numpy(), orc.lumped_H(nodes, tets, ref)) < 4e-7
