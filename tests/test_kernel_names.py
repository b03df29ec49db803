"""Which kernel an accumulate or a batched launch uses (host only)."""
import ctypes as C

import pytest

from paper_2111_10448_gb300 import _native as N

BF16, TF32, FP16, FP64 = N.TT_PREC_BF16, N.TT_PREC_TF32, N.TT_PREC_FP16, N.TT_PREC_FP64


def _problem(dims, r, p, prec, flags=0, passes=1):
    d = len(dims)
    return N.make_problem(dims, ranks=[1] + [r] * (d - 1) + [1], p=p, seed=1, passes=passes,
                          x_dtype=N.TT_F64 if prec == FP64 else N.TT_F32, prec=prec, flags=flags)


CASES = [
    ("fp64", [20, 20, 20], 4, 4, FP64, 0, 1),
    ("plane", [256, 6, 256], 6, 10, BF16, 0, 1),
    ("slab", [256, 4, 4, 256], 6, 10, FP16, N.TT_FLAG_KR, 1),
    ("strip", [40, 7, 6, 70], 4, 6, BF16, 0, 1),
    ("strip", [40, 7, 6, 70], 4, 6, TF32, N.TT_FLAG_KR, 1),
    ("strip", [24] * 6, 10, 16, BF16, 0, 1),            # small planes up to three sketches a side
    ("strip", [12, 5, 4, 12], 4, 4, FP16, 0, 1),
    ("small-plane", [12, 5, 4, 12], 4, 4, TF32, N.TT_FLAG_KR, 1),
    ("small-plane", [12] * 7, 4, 4, BF16, 0, 1),        # four on the column side
    ("tile", [40, 3, 3, 3, 3, 3, 40], 3, 4, BF16, 0, 1),
    ("tile", [40, 9, 8, 40], 4, 4, BF16, N.TT_FLAG_ONESIDED, 2),   # no sketch on the column side
    ("tile", [60, 70], 4, 4, BF16, 0, 2),
]


@pytest.mark.parametrize("name,dims,r,p,prec,flags,passes", CASES)
def test_single(name, dims, r, p, prec, flags, passes):
    L = N.lib()
    h = C.c_void_p()
    q = _problem(dims, r, p, prec, flags, passes)
    N.check(L.tt_sketch_plan(C.byref(q), C.byref(h)), "plan")
    assert L.tt_sketch_kernel_name(h, dims[-1]).decode() == name
    # the coarser numbering is as documented
    sp = name == "small-plane" or (name == "strip" and max(dims[0], dims[-1]) <= 32 and not flags & N.TT_FLAG_KR)
    kind = 3 if sp else {"fp64": 0, "plane": 2, "slab": 2, "strip": 1, "tile": 1}[name]
    assert L.tt_sketch_kernel_kind(h, dims[-1]) == kind
    L.tt_plan_destroy(h)


@pytest.mark.parametrize("name,shapes,prec", [
    ("fp64", [[8, 9, 8], [10] * 4], FP64),
    ("strip", [[8, 9, 8], [24] * 4, [9] * 6], BF16),
    ("small-plane", [[8, 9, 8], [24] * 4, [5] * 7], TF32),
    ("tile", [[8, 9, 8], [33, 5, 20]], FP16),
])
def test_batch(name, shapes, prec):
    L = N.lib()
    h = C.c_void_p()
    arr = (N.tt_problem * len(shapes))(*[_problem(d, 3, 4, prec) for d in shapes])
    N.check(L.tt_sketch_plan_batched(arr, len(shapes), C.byref(h)), "plan")
    assert L.tt_sketch_kernel_name(h, 0).decode() == name
    L.tt_plan_destroy(h)


def test_no_plan():
    assert N.lib().tt_sketch_kernel_name(C.c_void_p(0), 1) == b""
