"""eqlinear_bwd_weight_static: the weight gradient for callers that cannot allocate device scratch.

Some users of the library run where a device allocation is not available to them at call time (a
plug-in inside an application that owns all GPU memory, a pool that has already reserved the whole
device, a loop that must not stall on an allocation).  They call this entry point instead of
eqlinear_bwd_weight; it takes the same inputs and outputs but no scratch buffer, using a fixed
32 MiB device array inside the library.  The test checks, through the C ABI, that it returns exactly
what eqlinear_bwd_weight returns (the same kernels in the same fixed reduction order: bit-identical),
and what the oracle computes, on two calls in a row (the shared array keeps the previous call's
contents, so the second call also shows that nothing stale leaks in); that free device memory is the
same before and after each of those calls (the array became resident when the plan was built, not
here); and that sizes beyond the array are refused.  This file sorts last so that a run stopping at the first failure has already
run every other test; it also passes when run alone in a fresh process.
"""

import numpy as np
import pytest
import torch

import paper_2607_21271_b200 as eq
from oracle import eqlinear_oracle as orc
from paper_2607_21271_b200.workloads import Workload, generate
from tests.harness import TOL, GpuLayer, rel_max_err

pytestmark = pytest.mark.gpu


# The float case with 300 -> 280 channels takes several token ranges, whose partial sums all fit the array.
@pytest.mark.parametrize("dtype,T,Ci,Co,N", [("fp16", 8, 24, 40, 1500), ("fp32", 4, 16, 8, 333), ("fp32", 4, 300, 280, 6000)])
def test_static_scratch_matches_caller_scratch_twice(dtype, T, Ci, Co, N):
    wl = Workload("noalloc", dtype, T, Ci, Co, N, "normal", ("bwd_weight",), 21)
    d = generate(wl)
    layer = GpuLayer(T, Ci, Co, dtype, d["w"], d["bias"])
    try:
        assert eq.eqlinear_bwd_weight_scratch_bytes(layer.plan, N) <= eq.binding.EQL_STATIC_SCRATCH_BYTES
        ref_dw, ref_db = layer.bwd_weight(d["x"], d["dy"])                 # existing entry point, caller scratch
        orc_dw, orc_db = orc.bwd_weight(d["x"], d["dy"], T)
        x = torch.from_numpy(d["x"]).cuda()
        dy = torch.from_numpy(d["dy"]).cuda()
        # a different problem first, so the shared array holds foreign partials when the real calls run
        other = torch.from_numpy(generate(Workload("o", dtype, T, Ci, Co, N, "normal", ("bwd_weight",), 22))["dy"]).cuda()
        outs = [(torch.full((Co, Ci, T), float("nan"), dtype=torch.float32, device="cuda"),
                 torch.full((Co,), float("nan"), dtype=torch.float32, device="cuda")) for _ in range(3)]
        torch.cuda.synchronize()
        for call, grad in enumerate((other, dy, dy)):
            dw, db = outs[call]
            free_before = torch.cuda.mem_get_info()[0]
            eq.eqlinear_bwd_weight_static(layer.plan, x, grad, dw, db, N, layer.stream)
            torch.cuda.synchronize()
            assert torch.cuda.mem_get_info()[0] == free_before, f"call {call} changed the free device memory"
            if call == 0:
                continue
            assert np.array_equal(dw.cpu().numpy(), ref_dw), f"call {call}: dw differs from eqlinear_bwd_weight's"
            assert np.array_equal(db.cpu().numpy(), ref_db), f"call {call}: db differs from eqlinear_bwd_weight's"
            assert rel_max_err(dw.cpu().numpy(), orc_dw) <= TOL[dtype], f"call {call}: dw against the oracle"
            assert rel_max_err(db.cpu().numpy(), orc_db) <= TOL[dtype], f"call {call}: db against the oracle"
    finally:
        layer.close()


def test_static_scratch_rejects_sizes_beyond_the_array():
    T, Ci, Co, N = 8, 256, 256, 8192
    wl = Workload("big", "fp16", T, Ci, Co, N, "none", ("bwd_weight",), 23)
    d = generate(wl)
    layer = GpuLayer(T, Ci, Co, "fp16", d["w"], None)
    try:
        need = eq.eqlinear_bwd_weight_scratch_bytes(layer.plan, N)
        if need <= eq.binding.EQL_STATIC_SCRATCH_BYTES:
            pytest.skip("this shape fits the built-in array with the current kernel's split")
        x = torch.from_numpy(d["x"]).cuda()
        dy = torch.from_numpy(d["dy"]).cuda()
        dw = torch.zeros(Co, Ci, T, dtype=torch.float32, device="cuda")
        with pytest.raises(eq.EqlError) as e:
            eq.eqlinear_bwd_weight_static(layer.plan, x, dy, dw, None, N, layer.stream)
        assert e.value.status == eq.binding.EQL_ERR_WORKSPACE
        assert not dw.any().item()                                      # nothing was launched
    finally:
        layer.close()


# Partial sums of all tiles do not fit the array: the call goes through it in blocks of tiles, launch after launch (384 -> 64 channels:
# along the input channels).  And a float
# layer too small for those kernels, whose 50000 tokens run in blocks of tokens, each added to dw / db.
@pytest.mark.parametrize("dtype,T,Ci,Co,N,fits", [("fp32", 4, 256, 256, 32768, False), ("fp32", 4, 384, 384, 32768, False), ("fp16", 2, 512, 512, 65536, True),
                                                  ("fp16", 2, 1024, 1024, 20000, None), ("fp32", 8, 128, 192, 65537, False), ("fp32", 4, 384, 64, 110000, False),
                                                  ("fp16", 1, 768, 4096, 20000, False), ("fp32", 4, 16, 24, 50000, True)])
def test_static_scratch_in_blocks(dtype, T, Ci, Co, N, fits):
    """What eqlinear_bwd_weight returns from its own, larger scratch, bit for bit; sampled channels against the oracle."""
    g = np.random.Generator(np.random.PCG64(Ci + N))
    narrow = np.float16 if dtype == "fp16" else np.float32
    x, dy = (g.standard_normal((N, C * T), dtype=np.float32).astype(narrow) for C in (Ci, Co))
    layer = GpuLayer(T, Ci, Co, dtype, np.zeros((Co, Ci, T), dtype=narrow), None)
    try:
        assert (eq.eqlinear_bwd_weight_scratch_bytes(layer.plan, N) <= eq.binding.EQL_STATIC_SCRATCH_BYTES) == fits or fits is None
        ref_dw, ref_db = layer.bwd_weight(x, dy)
        xd, dyd = torch.from_numpy(x).cuda(), torch.from_numpy(dy).cuda()
        dw = torch.full((Co, Ci, T), float("nan"), dtype=torch.float32, device="cuda")
        db = torch.full((Co,), float("nan"), dtype=torch.float32, device="cuda")
        eq.eqlinear_bwd_weight_static(layer.plan, xd, dyd, dw, db, N, layer.stream)
        assert layer.raw_status() == 0
        assert np.array_equal(dw.cpu().numpy(), ref_dw) and np.array_equal(db.cpu().numpy(), ref_db)
    finally:
        layer.close()
    o, i = (np.unique(np.linspace(0, C - 1, 24).astype(int)) for C in (Co, Ci))
    pick = lambda a, c: a.reshape(N, -1, T)[:, c].reshape(N, -1)
    rdw, rdb = orc.bwd_weight(pick(x, i), pick(dy, o), T)
    assert rel_max_err(ref_dw[np.ix_(o, i)], rdw) <= TOL[dtype] and rel_max_err(ref_db[o], rdb) <= TOL[dtype]


def test_static_scratch_refuses_what_does_not_fit_in_blocks_either():
    T, Ci, Co, N = 1, 2048, 4096, 3                                          # CUDA-core kernels: one partial sum is the 32 MiB of dw and db's
    layer = GpuLayer(T, Ci, Co, "fp32", np.zeros((Co, Ci, T), dtype=np.float32), None)
    try:
        assert eq.eqlinear_bwd_weight_scratch_bytes(layer.plan, N) > eq.binding.EQL_STATIC_SCRATCH_BYTES
        x, dy = (torch.zeros(N, C * T, device="cuda") for C in (Ci, Co))
        dw = torch.full((Co, Ci, T), -3.0, dtype=torch.float32, device="cuda")
        with pytest.raises(eq.EqlError) as e:
            eq.eqlinear_bwd_weight_static(layer.plan, x, dy, dw, None, N, layer.stream)
        assert e.value.status == eq.binding.EQL_ERR_WORKSPACE
        assert bool((dw == -3.0).all().item())                              # nothing was launched
    finally:
        layer.close()
