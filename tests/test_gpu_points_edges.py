"""vfmm_evaluate_points where its closed forms change branch, with rough leaf values.

Odd and even k down to 4 (ragged classes of the leaf coefficients), a single leaf (no far field) and a
graded tree; points along a line off a leaf edge from 1e-14 of its width to half of it (the edge
recurrence turns from upwards to downwards at about 0.04), at and next to corners. Same bar as the other
tests of this entry point: 1e-12 of the largest value.
"""
import numpy as np
import pytest

import workloads as W
from oracle import offnode
from oracle import tree as T

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1610_00823_gb300 as v  # noqa: E402

TOL = 1e-12


@pytest.mark.parametrize("k,p,kind", [(4, 6, "leaf"), (11, 27, "leaf"), (5, 12, "graded"), (16, 40, "uniform")])
def test_points_near_edges_and_corners(k, p, kind, oracle_ops):
    if kind == "graded":
        src = W.narrow_gaussians(5, n=3, sigma=0.04)
        gt = v.tree_build(0.0, 0.0, 1.0, k, src, 1e-2, 5, min_depth=2)
        ot = T.build_adaptive(0.0, 0.0, 1.0, k, src, 1e-2, 5, min_depth=2)
        assert gt.list_len[2] > 0
    else:
        d = 0 if kind == "leaf" else 2
        gt = v.tree_build_uniform(0.0, 0.0, 1.0, k, d)
        ot = T.build_uniform(0.0, 0.0, 1.0, k, d)
    F = np.random.default_rng(k).standard_normal((ot.n_leaves, k * k))
    f = torch.from_numpy(F.reshape(-1)).cuda()
    ops = v.ops_create(k, p)
    ws = v.workspace(gt, ops, 1)
    v.volume_potential(gt, ops, f, ws=ws)
    b = int(ot.leaves[ot.n_leaves // 2])
    h = float(ot.h(b))
    cx, cy = ot.centre(b)
    off = np.array([1e-14, 1e-11, 1e-7, 1e-4, 1e-3, 0.01, 0.03, 0.037, 0.04, 0.043, 0.06, 0.1, 0.2, 0.4, 0.5])
    pts = [np.column_stack([cx - h / 2 + off * h, np.full(off.size, cy + 0.13 * h)]),
           np.column_stack([np.full(off.size, cx - 0.31 * h), cy + h / 2 - off * h]),
           np.column_stack([cx + h / 2 - off * h, cy - h / 2 + 0.7 * off * h]),
           np.array([[cx - h / 2, cy - h / 2], [cx - h / 2, cy + 0.2 * h], [cx, cy]])]
    pts = np.concatenate(pts)
    x, y = (torch.from_numpy(pts[:, i].copy()).cuda() for i in (0, 1))
    got = [o.cpu().numpy() for o in v.evaluate_points(gt, ops, f, ws, x, y)]
    ref = offnode.evaluate(ot, T.build_lists(ot), oracle_ops(k, p), F, pts[:, 0], pts[:, 1])
    for q in range(3):
        assert np.max(np.abs(got[q] - ref[q])) < TOL * np.max(np.abs(ref[q])), q
