"""Distinct M2L translations: offsets beyond the 19 packed bits take the host map.  Two cubes of side 2e-6
at distance 1.6 with theta = 3e-6 interact at levels 18 and 19, half a million half-cells apart.  M lives in
one cube alone, so u on the other is the far field; the recurrence per pair (no table, no keys) is the
reference.  FP64: rounding of ~1e3 terms, 1e-12; FP32 and split BF16: their bars elsewhere (2e-6, 3e-5)."""
import numpy as np
import pytest
import torch

from paper_1606_00247_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_wide_offsets_take_the_host_map():
    from paper_1606_00247_gb300.api import Plan

    cube, t = inputs.unit_cube(3)
    nodes = np.vstack([2e-6 * cube, np.array([1.0, 0.9, 0.8]) + 2e-6 * cube])
    tets = np.vstack([t, t + len(cube)]).astype(np.int32)
    M = inputs.gaussian_unit_m(len(nodes), batch=9, seed=21)
    M[:, : len(cube)] = 0.0
    Md = torch.as_tensor(M, device="cuda")
    kw = dict(p=4, leaf_size=8, theta=3e-6, near_mode=0, max_batch=9)

    def far(**o):
        return Plan(nodes, tets, **kw, **o).eval(Md)[0][:, : len(cube)].cpu().numpy()

    ex = Plan(nodes, tets, **kw).export_tree()
    k = np.zeros((len(ex["cell_level"]), 3), np.int64)  # box coordinates: x bits at 3b, y at 3b + 1, z at 3b + 2
    for b in range(21):
        k |= (((ex["cell_prefix"][:, None] >> np.uint64(3 * b) >> np.arange(3, dtype=np.uint64)) & np.uint64(1)) << np.uint64(b)
              ).astype(np.int64)
    tgt = np.repeat(np.arange(len(k)), np.diff(ex["m2l_off"]))
    same = ex["cell_level"][tgt] == ex["cell_level"][ex["m2l_src"]]
    off = 2 * (k[tgt] - k[ex["m2l_src"]])[same]
    assert len(tgt) > 50 and np.abs(off).max() >= 2**18  # not packable

    ref = far(precision="fp64", m2l_table_batch=-1)
    for prec, bar in (("fp64", 1e-12), ("fp32", 2e-6), ("bf16x3", 3e-5)):
        u = far(precision=prec)
        assert np.linalg.norm(u - ref) < bar * np.linalg.norm(ref), prec
