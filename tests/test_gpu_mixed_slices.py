"""The mixed form's accuracy by slice count, near and leaf far field in reflection classes (k >= 6).

* A leaf value below the last digit: S slices round an operand at 2^(-7 S - 1) of its power-of-two scale.
  Beside a value that sets the scale, in a leaf far away, a value of 0.75 units of 2^(-7 S) must come through
  to half a unit: the difference of two solves against the FP64 solve of that value alone. The neighbours'
  values are zero, so the value's orbits have this one member.
* S = 7 and 8 for all five contractions, rough values: the mixed form's bar of 1e-10 at S = 6 falls by 2^7
  with every slice, down to what the double-FP32 sums keep (at most 40 additions, rounded at 2^-48 each).
"""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1610_00823_gb300 as v  # noqa: E402


@pytest.mark.parametrize("k", [6, 7, 9, 16])
def test_value_below_the_last_digit(k):
    S = 6
    tree = v.tree_build_uniform(0.0, 0.0, 1.0, k, 3)
    p = int(2.5 * k)
    mixed = v.ops_create(k, p, v.MIXED)
    mixed.set_slices(near=S, s2m=8, m2l=8, s2l=8, far=8)
    kk = k * k
    x, y = (c.reshape(-1, kk) for c in tree.leaf_nodes())
    mid = lambda c: 0.5 * (c.amin(1) + c.amax(1))
    cx, cy = mid(x), mid(y)
    at = lambda px, py: int(((cx - px).abs() + (cy - py).abs()).argmin())
    big, small = at(0.44, 0.44), at(-0.31, -0.19)
    f = torch.zeros(tree.n_leaves, kk, dtype=torch.float64)
    f[big, kk // 2] = 1.0  # below 2^1: units of 2^(1 - 7 S)
    unit = 2.0 ** (1 - 7 * S)
    only = torch.zeros_like(f)
    only[small, (k // 3) * k + 1] = 0.75 * unit
    both = v.volume_potential(tree, mixed, (f + only).reshape(-1).cuda())
    without = v.volume_potential(tree, mixed, f.reshape(-1).cuda())
    ref = v.volume_potential(tree, v.ops_create(k, p), only.reshape(-1).cuda())
    torch.cuda.synchronize()
    for q in range(3):
        err = float(((both[q] - without[q]) - ref[q]).abs().max() / ref[q].abs().max())
        assert err <= 0.5 / 0.75 + 2.0 ** -4, (q, err)  # and the sums' own rounding


@pytest.mark.parametrize("k", [6, 9, 11, 16])
@pytest.mark.parametrize("S", [7, 8])
def test_more_slices(k, S):
    src = W.narrow_gaussians(5, n=3, sigma=0.04)
    tol = {6: 1e-3, 9: 1e-5, 11: 1e-6, 16: 1e-10}[k]
    tree = v.tree_build(0.1, -0.2, 1.5, k, src, tol, 6, min_depth=3)
    assert min(tree.list_len) > 0
    p = int(2.5 * k)
    mixed = v.ops_create(k, p, v.MIXED)
    mixed.set_slices(near=S, s2m=S, m2l=S, s2l=S, far=S)
    g = torch.Generator(device="cpu").manual_seed(k)
    f = torch.randn(tree.n_leaves * k * k, generator=g, dtype=torch.float64).cuda()
    got = v.volume_potential(tree, mixed, f)
    ref = v.volume_potential(tree, v.ops_create(k, p), f)
    torch.cuda.synchronize()
    for q in range(3):
        err = float((got[q] - ref[q]).abs().max() / ref[q].abs().max())
        assert err < 1e-10 * 2.0 ** (-7 * (S - 6)) + 40 * 2.0 ** -48, (q, err)
