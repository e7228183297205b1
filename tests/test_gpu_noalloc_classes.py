"""The allocation-free solve with the reflection-class contractions of the mixed form (k >= 6).

* Trees that its 32 MiB scratch held when near and leaf far field were gathered row by row stay accepted
  (the operand buffer takes what the rest leaves).
* Operand tiles in several chunks that end inside a group of leaves: at k = 16 three groups have some 800 tiles
  of 48 KB and the scratch room for about half of them; odd k makes its classes one by one. Against the
  workspace solve, which has one chunk: the same digits and products, double-FP32 sums in another order
  (K blocks shared by several CTAs), at most 40 additions rounded at 2^-48 in either.
"""
import ctypes

import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1610_00823_gb300 as v  # noqa: E402
from paper_1610_00823_gb300 import _lib  # noqa: E402

TOL = 2 * 40 * 2.0 ** -48


def _check(tree, ops):
    g = torch.Generator(device="cpu").manual_seed(tree.k)
    f = torch.randn(tree.n_leaves * tree.k ** 2, generator=g, dtype=torch.float64).cuda()
    want = v.volume_potential(tree, ops, f)
    out = tuple(torch.full_like(f, float("nan")) for _ in range(3))
    lib = _lib.load()
    rc = lib.vfmm_volume_potential_noalloc(tree.handle, ops.handle, ctypes.c_void_p(f.data_ptr()), 1,
                                           *[ctypes.c_void_p(o.data_ptr()) for o in out],
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, lib.vfmm_last_error_detail()
    torch.cuda.synchronize()
    assert lib.vfmm_workspace_status(None) == 0
    for q in range(3):
        assert float((out[q] - want[q]).abs().max() / want[q].abs().max()) < TOL, q


@pytest.mark.parametrize("k,p,leaves", [(6, 60, 300), (7, 60, 339), (8, 60, 300)])
def test_trees_accepted_before_stay_accepted(k, p, leaves):
    src = W.uniform_gauss3().sources[0]
    _check(v.tree_build_leaves(0.0, 0.0, 1.0, k, src, leaves), v.ops_create(k, p, v.MIXED))


@pytest.mark.parametrize("k,p,leaves", [(16, 40, 300), (16, 20, 361), (15, 37, 300), (13, 32, 420)])
def test_operand_in_chunks(k, p, leaves):
    src = W.narrow_gaussians(5, n=3, sigma=0.04)
    tree = v.tree_build_leaves(0.0, 0.0, 1.0, k, src, leaves)
    assert min(tree.list_len) > 0
    _check(tree, v.ops_create(k, p, v.MIXED))
