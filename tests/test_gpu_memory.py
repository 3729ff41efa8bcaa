"""Device memory of solvers, network read-back and plans."""
import ctypes
import glob
import os

import numpy as np
import pytest
import torch

import paper_2501_04684_gb300 as ie
import workloads as W
from gpu_util import dev, empty, host, rel_l2

pytestmark = pytest.mark.gpu


def _problem(n, nb, edge=4.0):
    g = W.rng(1000 + n)
    ijk = W.full_grid(n)
    counts = np.full(len(ijk), nb, np.int32)
    return W.Problem(name="memory", G=n, box_ijk=ijk, nb=counts, P=W.random_P(g, counts), alpha=W.alpha_for("tiny"), a=1.0 / edge)


def test_solver_footprint_counts_the_refinement():
    """A refined solve keeps, per unknown and column, an FP64 iterate and three FP32 vectors (40
    bytes), and one FP64 pair per chunk of 512 unknowns."""
    p, R = _problem(4, 20), 3
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_FP32), R)) as plan:
        plain = ie.ie_solver_footprint(plan.handle, R, ie.solve_opts())
        refined = ie.ie_solver_footprint(plan.handle, R, ie.solve_opts(refine=1))
        assert refined - plain == 40 * R * p.n + 16 * R * -(-p.n // 512)


def _pool_high(reset=False):
    """High-water mark of the device's stream-ordered pool, bytes in use (0 where it is unknown)."""
    rt = ctypes.CDLL(None)
    if not hasattr(rt, "cudaDeviceGetDefaultMemPool"):
        found = glob.glob(os.path.join(os.path.dirname(torch.__file__), "..", "nvidia", "**", "libcudart.so*"), recursive=True) + \
            glob.glob("/usr/local/cuda/lib64/libcudart.so*")
        rt = ctypes.CDLL(found[0])
    pool, v = ctypes.c_void_p(), ctypes.c_uint64()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    attr = 8                                            # cudaMemPoolAttrUsedMemHigh
    if reset:
        assert rt.cudaMemPoolSetAttribute(pool, attr, ctypes.byref(v)) == 0
    assert rt.cudaMemPoolGetAttribute(pool, attr, ctypes.byref(v)) == 0
    return v.value


def test_reading_networks_back_takes_a_bounded_scratch():
    p = W.Problem(name="nets", G=24, box_ijk=np.array([(x, y, z) for x in range(0, 24, 2) for y in (0, 3) for z in (0, 5)], np.int32),
                  nb=np.full(48, 2, np.int32), P=W.random_P(W.rng(1010), np.full(48, 2)), alpha=1.0)
    with ie.Plan(ie.problem_from(p, ie.precmask(ie.IE_PREC_CVFCNN_FP32), cvfcnn_hidden=64)) as plan:
        n = plan.stats["n_coupling_blocks"]
        assert n > 150
        g = W.rng(1011)
        w = [W.complex_normal(g, s).astype(np.complex64) for s in ((n, 64, 192), (n, 64), (n, 192, 64), (n, 192))]
        ie.ie_cvfcnn_set_weights(plan.handle, *w)
        _pool_high(reset=True)
        start = _pool_high()
        back = ie.ie_cvfcnn_get_weights(plan.handle)
        assert _pool_high() - start <= 16 << 20         # all of them take n * 198 KB
        for a, b in zip(w, back):
            assert np.array_equal(a, b)


def test_a_plan_that_fits_without_the_convolution_is_made_without_it():
    p = _problem(8, 64)
    mask = ie.precmask(ie.IE_PREC_FP32)
    with ie.Plan(ie.problem_from(p, mask, symmetry=1)) as plan:
        assert ie.ie_plan_far_bytes(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, 1) > 0
        with_conv = plan.stats["device_bytes"]
        c = dev(W.coefficients(p, 1, 1020))
        y = empty((1, p.n))
        ie.ie_matvec(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, c, y, 1)
        ref = host(y)
    q = _problem(8, 64, edge=16.0)                      # box edge lambda / 16: block products only
    with ie.Plan(ie.problem_from(q, mask, symmetry=1)) as plan:
        assert ie.ie_plan_far_bytes(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, 1) == 0
        without = plan.stats["device_bytes"]
    assert with_conv - without > 256 << 20
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    keep = without + (with_conv - without) // 2
    fill = torch.empty(free - keep, dtype=torch.uint8, device="cuda")
    try:
        with ie.Plan(ie.problem_from(p, mask, symmetry=1)) as plan:
            assert ie.ie_plan_far_bytes(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, 1) == 0
            y.zero_()
            ie.ie_matvec(plan.handle, ie.IE_FULL, ie.IE_PREC_FP32, c, y, 1)
            assert rel_l2(host(y), ref) <= 2e-6
    finally:
        del fill
        torch.cuda.empty_cache()
