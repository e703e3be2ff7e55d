"""GPU parity of the coset-split dense kernels at the edges of their tiles, against the float64 oracles."""

import numpy as np
import pytest
import torch

import paper_2607_21271_b200 as eq
from oracle import eqlinear_oracle as orc
from oracle import eqlinear_oracle_dihedral as dih
from tests.harness import TOL, GpuLayer, kernels_launched, rel_max_err
from paper_2607_21271_b200.workloads import round_to_bf16

pytestmark = pytest.mark.gpu

# (rotations, dihedral, C_in, C_out, tokens): pairs of token tiles are 256 rows, K stages 64 columns, column tiles 32 to
# 256, weight-gradient stages 64 tokens and tiles of whole channels inside 128 columns.
SHAPES = [
    (6, False, 4, 4, 1), (6, False, 92, 60, 257), (6, False, 44, 172, 640),        # one row; one row past a pair; 264 / 1032 columns
    (12, False, 2, 22, 63), (7, False, 8, 40, 65), (5, False, 56, 16, 255),        # unsplit: tuples that do not divide a tile
    (1, False, 8, 136, 129), (3, False, 88, 8, 5000),                              # narrow sides; token ranges
    (2, False, 36, 260, 511), (2, False, 4, 4, 70000),                             # pair distance 1
    (2, True, 6, 66, 300), (4, True, 17, 33, 1025), (8, True, 33, 9, 257),         # dihedral, even numbers of rotations
    (3, True, 4, 28, 65), (5, True, 12, 4, 200), (6, True, 2, 30, 333),            # dihedral, others
    (4, False, 18, 130, 513), (8, False, 65, 9, 96), (16, False, 33, 17, 255),     # pair distances 2, 4, 8, 16
    (32, False, 9, 35, 1030), (8, False, 32, 64, 40000), (4, False, 4, 248, 600),
]
# Float layers on these kernels: 33 to 768 columns per product, blocks of 16 columns, stages of 16 tokens, at most 80 per token
# range; weight gradients of at least 8192 entries per product.
SHAPES_F32 = [(4, 17, 3, 1), (4, 8, 192, 700), (8, 9, 6, 257), (4, 384, 24, 15), (8, 192, 191, 33), (4, 33, 125, 1281), (8, 40, 72, 6000)]


@pytest.mark.parametrize("dtype,T,dihedral,Ci,Co,N", [(d, *s) for s in SHAPES for d in ("fp16", "bf16")] +
                         [("fp32", T, False, *s) for T, *s in SHAPES_F32])
def test_split_kernels_match_oracle(dtype, T, dihedral, Ci, Co, N):
    """Every pass, twice (fixed reduction order: bit-identical).  The operands are rounded once more than the inputs at
    most (one sum of two; float: truncation of every addition to the accumulator, a third as many as there), so the bars of the
    frequency-domain kernels hold."""
    L = 2 * T if dihedral else T
    g = np.random.Generator(np.random.PCG64(1000 * T + Ci))
    narrow = {"fp16": lambda a: a.astype(np.float16), "bf16": round_to_bf16, "fp32": lambda a: a}[dtype]
    x, dy = (narrow(g.standard_normal((N, C * L), dtype=np.float32)) for C in (Ci, Co))
    w = narrow(g.standard_normal((Co, Ci, L), dtype=np.float32) / np.float32(np.sqrt(Ci * L)))
    b = narrow(g.standard_normal(Co, dtype=np.float32))
    layer = GpuLayer(T, Ci, Co, dtype, w, b, eq.EQL_FLAG_DIHEDRAL if dihedral else 0)
    try:
        y, dx = layer.fwd(x), layer.bwd_data(dy)
        dw, db = layer.bwd_weight(x, dy)
        assert np.array_equal(y, layer.fwd(x)) and np.array_equal(dx, layer.bwd_data(dy))
        dw2, db2 = layer.bwd_weight(x, dy)
        assert np.array_equal(dw, dw2) and np.array_equal(db, db2)
        assert layer.raw_status() == 0
        info = eq.eqlinear_plan_info(layer.plan)
        assert (info.fwd_kernel, info.bwd_data_kernel) == (4, 4)
        narrow_f32 = dtype == "fp32" and Ci * Co * L * L < 4 * 8192         # entries of dw's products: T / 2 channels' each
        assert info.bwd_weight_kernel == (1 if narrow_f32 else 4)
    finally:
        layer.close()
    ref = (dih.fwd(x, w, b, T), dih.bwd_data(dy, w, T), *dih.bwd_weight(x, dy, T)) if dihedral else \
          (orc.fwd(x, w, b), orc.bwd_data(dy, w), *orc.bwd_weight(x, dy, T))
    for name, got, want in zip(("y", "dx", "dw", "db"), (y, dx, dw, db), ref):
        assert rel_max_err(got, want) <= TOL[dtype], name


@pytest.mark.parametrize("flags", [0, eq.EQL_FLAG_CORRELATION])
@pytest.mark.parametrize("Ci,Co,N", [(64, 256, 1830), (64, 256, 1832), (96, 171, 1900), (300, 80, 1300), (104, 160, 24040)])
def test_wide_layers_of_order_8_match_oracle(Ci, Co, N, flags):
    """Plans that keep both sets of operands, on either side of the lines (N C_in C_out = 3e7, weight gradient 4e8): the resident
    kernel in one direction or both, output tiles and channel chunks that the layer does not fill."""
    g = np.random.Generator(np.random.PCG64(Ci + N))
    x, dy = (g.standard_normal((N, C * 8), dtype=np.float32).astype(np.float16) for C in (Ci, Co))
    w = (g.standard_normal((Co, Ci, 8), dtype=np.float32) / np.float32(np.sqrt(Ci * 8))).astype(np.float16)
    b = g.standard_normal(Co, dtype=np.float32).astype(np.float16)
    corr = flags != 0
    layer = GpuLayer(8, Ci, Co, "fp16", w, b, flags)
    try:
        y, dx, (dw, db) = layer.fwd(x), layer.bwd_data(dy), layer.bwd_weight(x, dy)
        assert layer.raw_status() == 0
    finally:
        layer.close()
    ref = (orc.fwd(x, w, b, corr), orc.bwd_data(dy, w, corr), *orc.bwd_weight(x, dy, 8, corr))
    for name, got, want in zip(("y", "dx", "dw", "db"), (y, dx, dw, db), ref):
        assert rel_max_err(got, want) <= TOL["fp16"], name


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("T,dihedral,Ci,Co,N", [(2, True, 10, 66, 300), (4, True, 17, 33, 1025), (8, True, 9, 33, 257), (2, False, 36, 260, 511)])
def test_inputs_of_unsplit_groups_are_not_rounded(dtype, T, dihedral, Ci, Co, N):
    """Dihedral groups, and the weight gradient of order 2, take 16-bit inputs and weights as they are, whatever half precision
    can hold: partners are above 32768 and of one sign, so that no two of them may be added in half precision.  y and dx are
    rounded once, by at most 2^-11 (2^-8 bfloat16) of a value; dw and db are float sums of exact products."""
    L = 2 * T if dihedral else T
    g = np.random.Generator(np.random.PCG64(77 * T + Ci))
    narrow = {"fp16": lambda a: a.astype(np.float16), "bf16": round_to_bf16}[dtype]

    def large(C):
        return narrow((g.uniform(35000, 60000, (N, C, L)) * g.choice([-1.0, 1.0], (N, C, 1))).reshape(N, C * L).astype(np.float32))

    x, dy = large(Ci), large(Co)
    w = narrow((0.01 * g.standard_normal((Co, Ci, L)) / np.sqrt(max(Ci, Co) * L)).astype(np.float32))
    layer = GpuLayer(T, Ci, Co, dtype, w, None, eq.EQL_FLAG_DIHEDRAL if dihedral else 0)
    try:
        got = dict(zip(("dw", "db"), layer.bwd_weight(x, dy)))
        if dihedral:                                                         # (the linear passes of order 2 transform their inputs)
            got["y"], got["dx"] = layer.fwd(x), layer.bwd_data(dy)
        assert layer.raw_status() == 0
    finally:
        layer.close()
    ref = {"y": dih.fwd(x, w, None, T), "dx": dih.bwd_data(dy, w, T)} if dihedral else {}
    ref["dw"], ref["db"] = (dih if dihedral else orc).bwd_weight(x, dy, T)
    for name, a in got.items():
        bar = TOL["fp32"] if name in ("dw", "db") else 1.01 * {"fp16": 2.0 ** -11, "bf16": 2.0 ** -8}[dtype]
        assert rel_max_err(a, ref[name]) <= bar, name


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("T,dihedral,Ci,Co,N", [(3, False, 128, 256, 12608), (4, True, 256, 128, 3000), (2, False, 192, 384, 12609), (12, False, 84, 42, 20000),
                                                (1, False, 64, 48, 70001)])
def test_weight_gradient_of_unsplit_groups_adds_as_accurately_as_floats(dtype, T, dihedral, Ci, Co, N):
    """The products are exact; the tensor core adds eight steps of 16 tokens with truncation, by at most 2^-23 and half of that on
    average each, before the sum is added to a rounded one: 8 x 2^-24 = 4.8e-7 of a partial sum, and some roundings of 6e-8."""
    L = 2 * T if dihedral else T
    g = np.random.Generator(np.random.PCG64(99 * T + Ci))
    narrow = {"fp16": lambda a: a.astype(np.float16), "bf16": round_to_bf16}[dtype]
    x, dy = (narrow(g.standard_normal((N, C * L), dtype=np.float32)) for C in (Ci, Co))
    w = narrow(np.zeros((Co, Ci, L), dtype=np.float32))
    layer = GpuLayer(T, Ci, Co, dtype, w, None, eq.EQL_FLAG_DIHEDRAL if dihedral else 0)
    try:
        dw, db = layer.bwd_weight(x, dy)
        again = layer.bwd_weight(x, dy)
        assert np.array_equal(dw, again[0]) and np.array_equal(db, again[1])
        assert layer.raw_status() == 0
    finally:
        layer.close()
    rdw, rdb = (dih if dihedral else orc).bwd_weight(x, dy, T)
    assert rel_max_err(dw, rdw) <= 8e-7 and rel_max_err(db, rdb) <= 8e-7


def test_float_layers_repeat_beside_other_work():
    """The float kernels' two groups of transform warps share the ring's slots: every call gives the same bits while another stream
    takes away memory bandwidth and time slots in varying amounts, and no bounded wait runs out."""
    T, Ci, Co, N = 8, 48, 64, 12608
    g = np.random.Generator(np.random.PCG64(5))
    x, dy = (g.standard_normal((N, C * T), dtype=np.float32) for C in (Ci, Co))
    w = g.standard_normal((Co, Ci, T), dtype=np.float32) / np.float32(np.sqrt(Ci * T))
    layer = GpuLayer(T, Ci, Co, "fp32", w, None)
    side = torch.cuda.Stream()
    noise = torch.zeros(1 << 26, device="cuda")
    try:
        first = (layer.fwd(x), layer.bwd_data(dy), *layer.bwd_weight(x, dy))
        for k in range(20):
            with torch.cuda.stream(side):
                for _ in range(1 + k % 4):
                    noise[: 1 << (18 + k % 9)].add_(1.0)
            for a, b in zip(first, (layer.fwd(x), layer.bwd_data(dy), *layer.bwd_weight(x, dy))):
                assert np.array_equal(a, b)
        assert layer.raw_status() == 0
    finally:
        layer.close()
    for a, b in zip(first, (orc.fwd(x, w, None), orc.bwd_data(dy, w), *orc.bwd_weight(x, dy, T))):
        assert rel_max_err(a, b) <= TOL["fp32"]


@pytest.mark.parametrize("dtype,T,Ci,Co,N", [("fp32", 4, 256, 256, 32768), ("fp16", 6, 92, 60, 5000)])
def test_scratch_below_the_stated_size_is_refused(dtype, T, Ci, Co, N):
    """The kernel, and with it the sums' order, depends on the plan and N only: less scratch than the plan asks for is an error."""
    layer = GpuLayer(T, Ci, Co, dtype, np.zeros((Co, Ci, T), dtype=np.float32), None)
    try:
        x, dy = (torch.zeros(N, C * T, dtype=layer.td, device="cuda") for C in (Ci, Co))
        dw = torch.full((Co, Ci, T), -3.0, dtype=torch.float32, device="cuda")
        need = eq.eqlinear_bwd_weight_scratch_bytes(layer.plan, N)
        scratch = torch.empty(need, dtype=torch.uint8, device="cuda")
        with pytest.raises(eq.EqlError) as e:
            eq.eqlinear_bwd_weight(layer.plan, x, dy, dw, None, N, scratch, need - 256, layer.stream)
        assert e.value.status == eq.binding.EQL_ERR_WORKSPACE
        assert bool((dw == -3.0).all().item())                              # nothing was launched
    finally:
        layer.close()


@pytest.mark.parametrize("dtype,T,Ci,Co,N", [("fp16", 8, 128, 144, 19969), ("bf16", 4, 256, 260, 10001), ("fp16", 16, 65, 40, 20000)])
def test_gelu_beside_a_long_reduction(dtype, T, Ci, Co, N):
    """Forward passes with GELU whose tiles are halved so that two accumulators are in flight: at least 16 stages of 32 representatives
    and several units per pair of SMs; columns that do not fill the last tile."""
    from scipy.special import erf
    g = np.random.Generator(np.random.PCG64(Ci))
    narrow = {"fp16": lambda a: a.astype(np.float16), "bf16": round_to_bf16}[dtype]
    x = narrow(g.standard_normal((N, Ci * T), dtype=np.float32))
    w = narrow(g.standard_normal((Co, Ci, T), dtype=np.float32) / np.float32(np.sqrt(Ci * T)))
    b = narrow(g.standard_normal(Co, dtype=np.float32))
    layer = GpuLayer(T, Ci, Co, dtype, w, b, eq.EQL_FLAG_GELU)
    try:
        y = layer.fwd(x)
        assert layer.raw_status() == 0
    finally:
        layer.close()
    ref = orc.fwd(x, w, b)
    assert rel_max_err(y, 0.5 * ref * (1.0 + erf(ref / np.sqrt(2.0)))) <= TOL[dtype]


@pytest.mark.parametrize("dtype,T,Ci,Co,N", [("fp16", 8, 96, 384, 197), ("bf16", 2, 8, 656, 72), ("fp16", 32, 9, 35, 300), ("fp16", 6, 92, 60, 257),
                                             ("bf16", 4, 18, 130, 513), ("fp32", 4, 16, 40, 300), ("fp32", 8, 24, 20, 700),
                                             ("fp16", 8, 96, 136, 19969), ("fp16", 8, 192, 136, 19969)])
def test_gelu_in_either_form_of_the_epilogue(dtype, T, Ci, Co, N):
    """Half group by half group (pair distances 1, 2, 4, 16 and unsplit, one unit per pair of SMs and several) and, from 24 stages of
    32 representatives on, unrolled (the last shape)."""
    from scipy.special import erf
    g = np.random.Generator(np.random.PCG64(Ci + N))
    narrow = {"fp16": lambda a: a.astype(np.float16), "bf16": round_to_bf16, "fp32": lambda a: a}[dtype]
    x = narrow(g.standard_normal((N, Ci * T), dtype=np.float32))
    w = narrow(g.standard_normal((Co, Ci, T), dtype=np.float32) / np.float32(np.sqrt(Ci * T)))
    b = narrow(g.standard_normal(Co, dtype=np.float32))
    for bias in (b, None):
        layer = GpuLayer(T, Ci, Co, dtype, w, bias, eq.EQL_FLAG_GELU)
        try:
            y = layer.fwd(x)
            assert layer.raw_status() == 0
        finally:
            layer.close()
        ref = orc.fwd(x, w, bias)
        assert rel_max_err(y, 0.5 * ref * (1.0 + erf(ref / np.sqrt(2.0)))) <= TOL[dtype]


@pytest.mark.parametrize("dtype,T,dihedral,Ci,Co,N,form", [
    ("fp16", 4, False, 128, 74, 1000, "<8, 16>"), ("bf16", 4, False, 128, 76, 1000, "<32, 8>"),      # 9472 and 9728 elements of four, 16 ranges
    ("fp16", 4, False, 64, 64, 1796, "<8, 16>"), ("fp16", 8, False, 60, 64, 1796, "<32, 8>"),        # 4096 and 7680, 29 and 19 ranges
    ("fp16", 4, False, 256, 256, 500, "<32, 8>"), ("fp16", 3, False, 128, 256, 1500, "<32, 8>"),     # wide layers with few ranges
    ("fp16", 6, False, 72, 72, 3000, "<32, 8>"), ("bf16", 4, True, 64, 64, 1000, "<8, 16>"),         # 7 and 8 ranges
    ("bf16", 8, False, 15, 24, 1500, "<8, 16>"), ("bf16", 8, False, 15, 24, 1796, "<32, 8>"),        # 47 and 57
    ("fp32", 4, False, 64, 64, 3000, "<32, 8>")])
def test_either_form_of_the_finalize_kernel(dtype, T, dihedral, Ci, Co, N, form):
    """The partial sums of dw are added by the form that was measured the faster one on either side of each line."""
    L = 2 * T if dihedral else T
    g = np.random.Generator(np.random.PCG64(Ci + N))
    narrow = {"fp16": lambda a: a.astype(np.float16), "bf16": round_to_bf16, "fp32": lambda a: a}[dtype]
    x, dy = (narrow(g.standard_normal((N, C * L), dtype=np.float32)) for C in (Ci, Co))
    w = narrow(g.standard_normal((Co, Ci, L), dtype=np.float32) / np.float32(np.sqrt(Ci * L)))
    layer = GpuLayer(T, Ci, Co, dtype, w, None, eq.EQL_FLAG_DIHEDRAL if dihedral else 0)
    try:
        dw, db = layer.bwd_weight(x, dy)
        names = [n for n in kernels_launched(lambda: layer.bwd_weight(x, dy)) if "finalize" in n]
        assert layer.raw_status() == 0
    finally:
        layer.close()
    ref = dih.bwd_weight(x, dy, T) if dihedral else orc.bwd_weight(x, dy, T)
    assert rel_max_err(dw, ref[0]) <= TOL[dtype] and rel_max_err(db, ref[1]) <= TOL[dtype]
    assert len(names) == 1 and "split_finalize_kernel" + form in names[0], names


@pytest.mark.parametrize("dtype,T,Ci,Co,N,form", [
    ("fp16", 8, 192, 768, 197, 1), ("bf16", 4, 384, 768, 197, 1), ("fp16", 16, 96, 192, 256, 1), ("bf16", 6, 256, 512, 197, 1),    # a unit per pair
    ("fp32", 8, 32, 32, 19969, 1), ("fp32", 4, 64, 40, 19969, 1),
    ("bf16", 2, 800, 132, 19969, 2), ("bf16", 4, 384, 260, 19969, 2), ("fp16", 8, 192, 65, 19969, 2), ("fp16", 16, 97, 40, 19969, 2),
    ("fp16", 32, 48, 35, 19969, 2), ("bf16", 32, 48, 35, 19969, 2), ("fp16", 6, 260, 60, 19969, 2), ("fp16", 2, 736, 132, 19969, 1)])    # 23 stages
def test_gelu_is_unrolled_where_a_long_main_loop_hides_it(dtype, T, Ci, Co, N, form):
    """From 24 stages and more than one unit per pair of SMs on; pair distances 1 to 16 and unsplit, both 16-bit types."""
    from scipy.special import erf
    g = np.random.Generator(np.random.PCG64(Ci + N))
    narrow = {"fp16": lambda a: a.astype(np.float16), "bf16": round_to_bf16, "fp32": lambda a: a}[dtype]
    x = narrow(g.standard_normal((N, Ci * T), dtype=np.float32))
    w = narrow(g.standard_normal((Co, Ci, T), dtype=np.float32) / np.float32(np.sqrt(Ci * T)))
    b = narrow(g.standard_normal(Co, dtype=np.float32))
    layer = GpuLayer(T, Ci, Co, dtype, w, b, eq.EQL_FLAG_GELU)
    try:
        y = layer.fwd(x)
        names = [n for n in kernels_launched(lambda: layer.fwd(x)) if "linear" in n]
        assert layer.raw_status() == 0
    finally:
        layer.close()
    ref = orc.fwd(x, w, b)
    assert rel_max_err(y, 0.5 * ref * (1.0 + erf(ref / np.sqrt(2.0)))) <= TOL[dtype]
    assert len(names) == 1 and "split_linear_kernel<" in names[0] and f", {form}>" in names[0], names
