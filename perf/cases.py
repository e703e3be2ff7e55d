"""Performance cases of the equivariant linear layer: what programs that use the library have it do.

A case is one layer (group, channels per group element, data type), a number of tokens and what is done with them:

  "fwd"   inference: one forward call with fixed weights, optionally with the fused GELU;
  "step"  training: what one optimiser step does with the layer - take the new weight (eqlinear_plan_set_weight),
          forward, gradient of the input, gradient of weight and bias.  With "save" the forward pass keeps the spectrum
          of its input for the weight gradient (16-bit plans, as bench.py's headline step does).

Shapes are those of the package's workloads (token shapes of ViT and Swin at 224 x 224, the group-order sweep, the
operator-benchmark shapes) and, for the groups no workload names, generic ones.
"""

import torch

import paper_2607_21271_b200 as eq

DTYPES = {"fp32": (eq.EQL_FP32, torch.float32), "fp16": (eq.EQL_FP16, torch.float16), "bf16": (eq.EQL_BF16, torch.bfloat16)}
SPECTRUM_ORDERS = (4, 8, 16, 32)          # cyclic orders whose 16-bit plans have the saved-spectrum path


def _case(name, group, T, Ci, Co, N, dtype, mode, bias=True, gelu=False, save=False):
    c = {"group": group, "T": T, "Ci": Ci, "Co": Co, "N": N, "dtype": dtype, "mode": mode, "bias": bias, "gelu": gelu, "save": save}
    return {"name": name, **c} if name else c


def listed():
    return [
        # The smallest configuration of the package: nothing but the latency of a call.
        _case("tiny_fp32_fwd", "cyclic", 4, 8, 8, 64, "fp32", "fwd", bias=False),
        # Serving one image: the first MLP layer of a ViT-B block with its GELU, 197 tokens.
        _case("vit_b_fc1_one_image", "cyclic", 8, 96, 384, 197, "fp16", "fwd", gelu=True),
        # Training a ViT-S projection in single precision, batch 64 (12608 tokens).
        _case("vit_s_fp32_step", "cyclic", 8, 48, 48, 64 * 197, "fp32", "step"),
        # Training the widening MLP layer of ViT-B in half precision, batch 128: the headline layer of the benchmark.
        _case("vit_b_fc1_fp16_step", "cyclic", 8, 96, 384, 128 * 197, "fp16", "step", save=True),
        # The narrowing MLP layer of the same block in bfloat16: few outputs, long reduction.
        _case("vit_b_fc2_bf16_step", "cyclic", 8, 384, 96, 128 * 197, "bf16", "step"),
        # Inference on high-resolution windows: first stage of Swin-T, batch 128; memory traffic dominates.
        _case("swin_t_s1_fp16_fwd", "cyclic", 4, 24, 96, 128 * 56 * 56, "fp16", "fwd"),
        # Fine rotation groups at a constant total width of 1024 (the group-order sweep).
        _case("sweep_T16_fp16_step", "cyclic", 16, 64, 64, 65536, "fp16", "step"),
        _case("sweep_T32_fp16_step", "cyclic", 32, 32, 32, 65536, "fp16", "step"),
        # The operator benchmark's wide layer (total width 4096): the largest, bound by arithmetic.
        _case("op_c1024_fp16_step", "cyclic", 4, 1024, 1024, 32 * 1024, "fp16", "step"),
        # The operator benchmark in single precision (total width 1024).
        _case("op_c256_fp32_step", "cyclic", 4, 256, 256, 32 * 1024, "fp32", "step"),
        # Sixfold rotations (hexagonal lattices), a ragged number of tokens and uneven channels.
        _case("p6_fp16_step", "cyclic", 6, 92, 60, 10007, "fp16", "step"),
        # Rotations and reflections of the square: a ViT-sized layer over the dihedral group of order 8, batch 64.
        _case("d4_fp16_step", "dihedral", 4, 48, 96, 64 * 197, "fp16", "step"),
    ]


def _spread(rng, low, high):
    """A whole number from low to high, spread evenly over its logarithm."""
    return max(low, min(high, round(low * (high / low) ** rng.random())))


def draw(rng):
    kind = rng.choices(["T4_T8_16", "T2_T16_T32_16", "T4_T8_fp32", "other", "dihedral"], [9, 4, 3, 2, 2])[0]
    half = rng.choice(["fp16", "bf16"])
    group = "dihedral" if kind == "dihedral" else "cyclic"
    if kind == "T4_T8_16":
        T, dtype = rng.choice([4, 8]), half
    elif kind == "T2_T16_T32_16":
        T, dtype = rng.choice([2, 16, 32]), half
    elif kind == "T4_T8_fp32":
        T, dtype = rng.choice([4, 8]), "fp32"
    elif kind == "other":
        dtype = rng.choice([half, half, "fp32"])
        T = rng.choice([1, 3, 5, 6, 7, 12] + ([2, 16, 32] if dtype == "fp32" else []))
    else:
        T, dtype = rng.choice([2, 3, 4, 5, 6, 8]), rng.choice([half, half, "fp32"])
    tensor_cores = kind in ("T4_T8_16", "T2_T16_T32_16", "T4_T8_fp32")
    tuple_ = 2 * T if group == "dihedral" else T
    size = DTYPES[dtype][1].itemsize
    step = 1
    while (step * tuple_ * size) % 16:        # rows are whole 16-byte pieces: the only rule on channel counts
        step += 1
    top = 4096 // tuple_ if dtype != "fp32" and tensor_cores else 1024 // tuple_
    Ci, Co = (max(step, _spread(rng, 4, max(8, top)) // step * step) for _ in range(2))
    mode = rng.choice(["fwd", "step"])
    case = _case(None, group, T, Ci, Co, 1, dtype, mode, bias=rng.random() < 0.75,
                 gelu=mode == "fwd" and dtype != "fp32" and rng.random() < 0.3,
                 save=mode == "step" and dtype != "fp32" and group == "cyclic" and T in SPECTRUM_ORDERS and rng.random() < 0.5)
    # no more than the largest listed case costs: about 1 GB of tensors and its arithmetic, at the lower rates of single
    # precision and of the groups whose kernels do not run on the tensor cores
    w = work(case)
    flops = (16e9 if not tensor_cores else 75e9 if dtype == "fp32" else 800e9)
    most = min(400_000, int(1e9 / (2 * (Ci + Co) * tuple_ * size)), int(flops / w["flops"]))
    case["N"] = _spread(rng, 16, max(16, most))
    return case


class _State:
    """What a program holds for one layer: the plan with its workspace, parameters, activations and gradient buffers."""

    def __init__(self, case, seed):
        dtype, td = DTYPES[case["dtype"]]
        T, Ci, Co, N = case["T"], case["Ci"], case["Co"], case["N"]
        tuple_ = 2 * T if case["group"] == "dihedral" else T
        flags = (eq.EQL_FLAG_DIHEDRAL if case["group"] == "dihedral" else 0) | (eq.EQL_FLAG_GELU if case["gelu"] else 0)
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)

        def normal(*shape, std=1.0):
            return (torch.randn(*shape, generator=g, device="cuda") * std).to(td)

        def empty(*shape, like=td):
            return torch.empty(*shape, dtype=like, device="cuda")

        self.mode, self.save, self.N = case["mode"], case["save"], N
        self.stream = torch.cuda.current_stream().cuda_stream
        self.x = normal(N, Ci * tuple_)
        self.w = normal(Co, Ci, tuple_, std=(Ci * tuple_) ** -0.5)
        self.bias = normal(Co, std=0.02 ** 0.5) if case["bias"] else None
        self.y = empty(N, Co * tuple_)
        bytes_ = eq.eqlinear_workspace_bytes_flags(T, Ci, Co, dtype, flags)
        self.workspace = empty(bytes_, like=torch.uint8)
        self.plan = eq.eqlinear_plan(T, Ci, Co, dtype, self.w, self.bias, self.workspace, bytes_, flags=flags, stream=self.stream)
        if self.mode == "step":
            self.dy = normal(N, Co * tuple_)
            self.dx = empty(N, Ci * tuple_)
            self.dw = empty(Co, Ci, tuple_, like=torch.float32)
            self.db = empty(Co, like=torch.float32)
            self.scratch_bytes = eq.eqlinear_bwd_weight_scratch_bytes(self.plan, N)
            self.scratch = empty(max(256, self.scratch_bytes), like=torch.uint8)
            if self.save:
                self.spectrum_bytes = eq.eqlinear_spectrum_bytes(self.plan, N)
                self.spectrum = empty(self.spectrum_bytes, like=torch.uint8)

    def __del__(self):
        if getattr(self, "plan", None):
            eq.eqlinear_plan_destroy(self.plan)


def prepare(case, seed):
    return _State(case, seed)


def run(s):
    if s.mode == "fwd":
        eq.eqlinear_fwd(s.plan, s.x, s.y, s.N, stream=s.stream)
        return s.y
    eq.eqlinear_plan_set_weight(s.plan, s.w, s.bias, stream=s.stream)
    if s.save:
        eq.eqlinear_fwd_save_spectrum(s.plan, s.x, s.y, s.N, s.spectrum, s.spectrum_bytes, stream=s.stream)
    else:
        eq.eqlinear_fwd(s.plan, s.x, s.y, s.N, stream=s.stream)
    eq.eqlinear_bwd_data(s.plan, s.dy, s.dx, s.N, stream=s.stream)
    if s.save:
        eq.eqlinear_bwd_weight_from_spectrum(s.plan, s.spectrum, s.spectrum_bytes, s.dy, s.dw, s.db, s.N,
                                             s.scratch, s.scratch_bytes, stream=s.stream)
    else:
        eq.eqlinear_bwd_weight(s.plan, s.x, s.dy, s.dw, s.db, s.N, s.scratch, s.scratch_bytes, stream=s.stream)
    return {"y": s.y, "dx": s.dx, "dw": s.dw, "db": s.db}


def work(case):
    """Each tensor moved once, and the products of the fully block-diagonalised layer (one per real plane or
    one-dimensional representation, four per complex frequency, eight per two-dimensional representation)."""
    T, N, size = case["T"], case["N"], DTYPES[case["dtype"]][1].itemsize
    even = T % 2 == 0
    if case["group"] == "dihedral":
        tuple_, products = 2 * T, (4 * T - 4 if even else 4 * T - 2)
    else:
        tuple_, products = T, (1 if T == 1 else 2 * T - 2 if even else 2 * T - 1)
    params = case["Ci"] * case["Co"] * tuple_
    acts = N * (case["Ci"] + case["Co"]) * tuple_
    flops = 2.0 * products * N * case["Ci"] * case["Co"]
    if case["mode"] == "fwd":
        return {"bytes": float(acts * size + params * size), "flops": flops}
    return {"bytes": float(2 * acts * size + params * (size + 4)), "flops": 3 * flops}


def tolerance(case):
    """Two correct implementations differ by the roundings of operands and results to the data type: a few unit
    roundoffs (2^-11 for half precision, 2^-9 for bfloat16); single precision by the order of its sums."""
    return {"rel": {"fp32": 1e-5, "fp16": 2e-3, "bf16": 1e-2}[case["dtype"]]}
