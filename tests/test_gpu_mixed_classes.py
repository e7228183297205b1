"""The mixed form's near field in reflection classes, where its tiles and classes are ragged.

k from the smallest that takes this path (6) to 16, odd ones with a middle line; trees whose leaf count is no
multiple of the 128 leaves of a group, with every kind of orbit and operand tiles in several chunks
(graded), and several right-hand sides folded into a group; every slice count. Rough leaf values, against
the FP64 form at the mixed form's bar of 1e-10.
"""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1610_00823_gb300 as v  # noqa: E402

TOL = 1e-10


def _check(tree, k, nrhs, slices=6):
    p = int(2.5 * k)
    g = torch.Generator(device="cpu").manual_seed(k)
    f = torch.randn(nrhs * tree.n_leaves * k * k, generator=g, dtype=torch.float64).cuda()
    mixed = v.ops_create(k, p, v.MIXED)
    mixed.set_slices(near=slices)
    got = v.volume_potential(tree, mixed, f)
    ref = v.volume_potential(tree, v.ops_create(k, p), f)
    torch.cuda.synchronize()
    for q in range(3):
        err = float((got[q] - ref[q]).abs().max() / ref[q].abs().max())
        assert err < TOL, (q, err)


@pytest.mark.parametrize("k", [6, 7, 8, 11, 16])
def test_graded_tree(k):
    src = W.narrow_gaussians(5, n=3, sigma=0.04)
    tol = {6: 1e-3, 7: 1e-4, 8: 1e-5, 11: 1e-6, 16: 1e-10}[k]
    tree = v.tree_build(0.1, -0.2, 1.5, k, src, tol, 6, min_depth=3)
    assert min(tree.list_len) > 0 and tree.n_leaves % 128
    _check(tree, k, 1)


@pytest.mark.parametrize("k,depth,nrhs,slices", [(9, 3, 3, 6), (13, 2, 5, 7), (16, 3, 1, 8), (6, 0, 1, 6), (15, 1, 2, 6)])
def test_uniform_tree_folded_right_hand_sides(k, depth, nrhs, slices):
    _check(v.tree_build_uniform(0.1, -0.2, 1.5, k, depth), k, nrhs, slices)
