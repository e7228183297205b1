"""vfmm_evaluate_points next to a leaf corner, closer than the squares of the distances can hold.

The root box is centred at the origin, a corner of four leaves, where coordinates of any magnitude are
representable. u and its gradient are continuous there, with differences of about r log r: at 1e-150 and
below no result can be told from the one at the corner, up to the bar of the entry point's other tests (1e-12
of the largest value).
"""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1610_00823_gb300 as v  # noqa: E402

TOL = 1e-12


@pytest.mark.parametrize("k,p,graded", [(4, 10, False), (5, 12, True), (16, 40, False)])
def test_points_beside_a_corner(k, p, graded):
    if graded:  # leaves of two sizes meet at the origin
        tree = v.tree_build(0.0, 0.0, 1.0, k, W.narrow_gaussians(5, n=3, sigma=0.04), 1e-2, 5, min_depth=2)
    else:
        tree = v.tree_build_uniform(0.0, 0.0, 1.0, k, 2)
    g = torch.Generator(device="cpu").manual_seed(k)
    f = torch.randn(tree.n_leaves * k * k, generator=g, dtype=torch.float64).cuda()
    ops = v.ops_create(k, p)
    ws = v.workspace(tree, ops, 1)
    v.volume_potential(tree, ops, f, ws=ws)
    r = [1e-150, 1e-154, 1e-155, 1e-160, 1e-200, 1e-300, 5e-324]
    pts = [(0.0, 0.0)]
    for a in r:
        for sx in (-1, 0, 1):
            for sy in (-1, 0, 1):
                pts.append((sx * a, sy * a))
                pts.append((sx * a, sy * 1e-130))
                pts.append((sx * 1e-100, sy * a))
    x = torch.tensor([q[0] for q in pts], dtype=torch.float64).cuda()
    y = torch.tensor([q[1] for q in pts], dtype=torch.float64).cuda()
    far = torch.tensor([0.31], dtype=torch.float64).cuda()
    got = v.evaluate_points(tree, ops, f, ws, x, y)
    ref = v.evaluate_points(tree, ops, f, ws, far, far)  # another magnitude of the solution
    torch.cuda.synchronize()
    for q in range(3):
        assert torch.isfinite(got[q]).all(), q
        big = max(float(got[q][0].abs()), float(ref[q].abs().max()))
        assert float((got[q] - got[q][0]).abs().max()) < TOL * big, q
