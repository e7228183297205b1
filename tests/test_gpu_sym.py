"""The FP64 form's table products in reflection classes, at the sizes where classes are ragged.

Odd k has nodes on the axes (classes of unequal size, columns folded onto a middle line), p = 1 the
fewest parts per class, p = 60 the most; small trees leave most orbits with one entry, the graded tree
has every kind of list entry. Same bar as the other FP64 parity tests.
"""
import numpy as np
import pytest

import workloads as W
from oracle import fmm
from oracle import tree as T

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1610_00823_gb300 as v  # noqa: E402

TOL = 1e-13


@pytest.mark.parametrize("k,p", [(4, 1), (5, 7), (7, 60), (11, 27), (13, 24), (16, 47)])
@pytest.mark.parametrize("kind", ["uniform1", "uniform3", "graded"])
def test_fp64_solve_matches_oracle(k, p, kind, oracle_ops):
    src = W.narrow_gaussians(5, n=3, sigma=0.04)
    if kind == "graded":
        tol = {4: 1e-2, 5: 1e-2, 7: 1e-4, 11: 1e-6, 13: 1e-8, 16: 1e-10}[k]
        gt = v.tree_build(0.1, -0.2, 1.5, k, src, tol, 6, min_depth=3)
        ot = T.build_adaptive(0.1, -0.2, 1.5, k, src, tol, 6, min_depth=3)
        assert gt.n_leaves == ot.n_leaves and min(gt.list_len) > 0
    else:
        d = int(kind[-1])
        gt = v.tree_build_uniform(0.1, -0.2, 1.5, k, d)
        ot = T.build_uniform(0.1, -0.2, 1.5, k, d)
    # values without any symmetry: every class of every table is exercised
    F = np.random.default_rng(k * 100 + p).standard_normal((ot.n_leaves, k * k))
    u = v.volume_potential(gt, v.ops_create(k, p), torch.from_numpy(F.reshape(-1)).cuda())
    torch.cuda.synchronize()
    ref = fmm.solve(ot, T.build_lists(ot), oracle_ops(k, p), F)
    for q in range(3):
        got = u[q].cpu().numpy().reshape(ref[q].shape)
        assert np.max(np.abs(got - ref[q])) < TOL * np.max(np.abs(ref[q])), q


@pytest.mark.parametrize("k,p", [(5, 12), (8, 20), (16, 40)])
def test_workspace_is_no_larger_than_one_row_per_list_entry(k, p):
    """The allocation-free entry point takes what fits its scratch: a row per instance must not need
    more than a row per list entry did."""
    src = W.narrow_gaussians(5, n=3, sigma=0.02, spread=0.45)
    trees = [v.tree_build_uniform(0.0, 0.0, 1.0, k, d) for d in (2, 3, 5)]
    trees += [v.tree_build(0.0, 0.0, 1.0, k, src, 10.0 ** (1.0 - 0.6 * k), 8),
              v.tree_build_leaves(0.0, 0.0, 1.0, k, src, 200)]
    ops = v.ops_create(k, p)
    for t in trees:
        n_u, n_v, _, n_x = t.list_len
        rows = 8 * (3 * k * k * (n_u + t.n_leaves) + 2 * (p + 1) * (n_v + n_x + 2 * t.n_boxes))
        assert v.workspace_size(t, ops) <= rows + 4096 + 16 * t.n_boxes
