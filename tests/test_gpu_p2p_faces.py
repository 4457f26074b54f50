"""The integrated FP64 near field by faces of tet clusters (near_mode 0): the
affine functions of the two tets sharing a face differ by the jump of dM/dn alone,
a boundary face of a cluster takes the whole sum.  theta -> 0 makes every interaction
near field, so u is the oracle's direct sum (tet by tet, no sharing); 1e-12 as in
test_gpu_p2p_fp64."""
import numpy as np
import pytest
import torch

from paper_1606_00247_gb300 import inputs

pytestmark = pytest.mark.gpu


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _u(nodes, tets, M, **kw):
    from paper_1606_00247_gb300.api import Plan

    plan = Plan(nodes, tets, precision="fp64", near_mode=0, theta=1e-9, max_batch=M.shape[0], **kw)
    return plan.eval(torch.as_tensor(M, device="cuda"))[0].cpu().numpy()


# leaves of one tet (nothing shared) to one leaf cut into clusters of at most 40, and batches that
# take one slice, two, and a slice within a larger one
@pytest.mark.parametrize("B", [1, 4, 5, 19])
@pytest.mark.parametrize("leaf", [1, 6, 40, 41, 100000])
def test_clusters_vs_direct_sum(orc, leaf, B):
    nodes, tets = inputs.sphere(h=0.3)
    M = inputs.gaussian_unit_m(nodes.shape[0], batch=B, seed=77)
    u = _u(nodes, tets, M, p=1, leaf_size=leaf)
    for k in {0, B - 1}:
        assert rel_l2(u[k], orc.direct(nodes, tets, M[k])) < 1e-12


def test_single_tet_and_flat_cells(orc):
    nodes, tets = inputs.thin_film(6, 3, 2, size=(2000.0, 1000.0, 100.0))
    M = inputs.gaussian_unit_m(nodes.shape[0], batch=2)
    u = _u(nodes, tets, M, p=1, leaf_size=50)
    assert rel_l2(u[1], orc.direct(nodes, tets, M[1])) < 1e-12
    x = np.array([[0.0, 0.0, 0.0], [1.0, 0.0, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0], [3.0, 1.0, 0.5]])
    t = np.array([[0, 1, 2, 3]], dtype=np.int32)
    M = inputs.gaussian_unit_m(5, batch=1)
    assert rel_l2(_u(x, t, M, p=1, leaf_size=1)[0], orc.direct(x, t, M[0])) < 1e-12


def test_overlapping_tets_are_summed(orc):
    """A tet listed three times, and one laid over its neighbour on the same side of their
    face: the faces these share are no interior faces."""
    nodes, tets = inputs.sphere(h=0.45)
    a = tets[0]
    centre = nodes[tets[:, :]].mean(1)[0]
    nodes = np.vstack([nodes, nodes[a[:3]].mean(0) + 0.4 * (centre - nodes[a[:3]].mean(0))])
    over = np.array([[a[0], a[1], a[2], nodes.shape[0] - 1]], dtype=np.int32)  # inside tet 0, on its face
    t = np.concatenate([tets, tets[3:4], tets[3:4], over]).astype(np.int32)
    M = inputs.gaussian_unit_m(nodes.shape[0], batch=1, seed=5)
    u = _u(nodes, t, M, p=1, leaf_size=100000)
    assert rel_l2(u[0], orc.direct(nodes, t, M[0])) < 1e-12


# blocks of 4, 8 and 16 targets (by the share of the mesh a leaf's 16 nodes are), remainders in all;
# the stored near field integrates tet by tet, the far field is the same
@pytest.mark.parametrize("n, leaf", [(18, 20), (24, 32), (30, 32)])
def test_block_sizes_vs_stored(n, leaf):
    from paper_1606_00247_gb300.api import Plan

    nodes, tets = inputs.unit_cube(n)
    M = torch.as_tensor(inputs.gaussian_unit_m(nodes.shape[0], batch=2, seed=n), device="cuda")
    u = [Plan(nodes, tets, precision="fp64", near_mode=k, theta=0.5, p=3, leaf_size=leaf, max_batch=2)
         .eval(M)[0].cpu().numpy() for k in (0, 1)]
    assert rel_l2(u[0], u[1]) < 1e-12


def _film(ratio):  # cells of 333 x 333 and 333 / ratio
    return inputs.thin_film(6, 3, 2, size=(2000.0, 1000.0, 2.0 * 1000.0 / (3.0 * ratio)))


# Flattened and stretched tets, smooth M: no term of the face form is divided by a height of a triangle,
# so it is as accurate as the tet by tet form.  `stored`: the error of the stored coefficients (that form)
# against 80-bit arithmetic for these meshes and this M; the bar is four times that, as both results carry
# an error of its own.  (Face charges n.M instead: 1.2e-14, 3.7e-14, 4.9e-13, 1.6e-14 and 5.4e-14.)
@pytest.mark.parametrize("mesh, stored", [
    (lambda: _film(6.67), 1.65e-15), (lambda: _film(20.0), 3.97e-15), (lambda: _film(100.0), 1.72e-14),
    (lambda: inputs.sphere(h=0.3, scale=(1.0, 1.0, 0.05)), 3.17e-15),
    (lambda: inputs.sphere(h=0.3, scale=(1.0, 1.0, 20.0)), 3.63e-15)], ids=["film7", "film20", "film100", "disc", "needle"])
def test_flattened_tets_smooth_m(mesh, stored):
    from paper_1606_00247_gb300.api import Plan

    nodes, tets = mesh()
    r = np.random.default_rng(3)
    x = (nodes - nodes.mean(0)) / np.ptp(nodes, axis=0).max()
    M = sum(r.standard_normal(3) * np.cos(x @ (6.0 * r.standard_normal(3)) + 6.3 * r.random())[:, None] for _ in range(4))
    M = torch.as_tensor((M / np.linalg.norm(M, axis=1, keepdims=True))[None], device="cuda")
    for leaf in (4, 64):
        u = [Plan(nodes, tets, precision="fp64", near_mode=k, theta=1e-9, p=1, leaf_size=leaf).eval(M)[0].cpu().numpy()
             for k in (0, 1)]
        assert rel_l2(u[0], u[1]) < 4.0 * stored
