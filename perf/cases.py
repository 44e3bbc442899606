"""The work that users of this library have it do, as measurable cases.

Kinds of work:
  step      projections of a fine-tuned model: forward, backward through the frozen weight, LoRA gradients
            (or the forward alone); `layers` independent projections of one shape per pass
  block     the seven projections of a decoder block (q, k, v, o; gate, up; down), chained: forward only (token
            generation and evaluation) or forward and backward (fine-tuning)
  loss      the KL + cross-entropy loss of the error correction and its gradient
  quantize  min-max round-to-nearest quantization of one weight matrix

Weights are N(0, 0.02) quantized on the device by the library, adapters and activations as in the benchmark
configurations: A ~ U(-1/sqrt(K), 1/sqrt(K)), B ~ N(0, 0.01), X and dY ~ N(0, 1).
"""
import math

import torch

import paper_2306_08162_b200 as ql

BLOCK = (("q", 1, 1), ("k", 1, 1), ("v", 1, 1), ("o", 1, 1), ("gate", 1, 2), ("up", 1, 2), ("down", 2, 1))   # 1: hidden, 2: inner
BITS = (2, 3, 4, 8)


def step(name, **kw):
    case = dict(name=name, kind="step", bits=4, group=128, K=4096, N=4096, r=8, M=2048, layers=1, backward=True, dropout=0.0,
                act_order=False)
    case.update(kw)
    return case


def listed():
    return [
        # The smallest layer (512 x 512, 64 tokens): launches and latency are all there is.
        step("step_int4_512_m64", K=512, N=512, M=64),
        # Generating one token with the adapters attached: every projection of a block once, 100 MB of weights read.
        dict(name="decode_int4_m1", kind="block", bits=4, group=128, hidden=4096, inner=11008, r=8, M=1, backward=False),
        # A handful of tokens per step, one projection in each of 32 layers (together larger than the L2 cache).
        step("step_int3_m16_x32", bits=3, M=16, layers=32),
        # A short sequence, 8-bit weights.
        step("step_int8_m128", bits=8, M=128),
        # A ragged number of tokens through a fine-grained activation-order checkpoint (group 32), MLP down projection.
        step("step_int4_g32_actorder_m333", group=32, K=11008, N=4096, M=333, act_order=True),
        # The usual fine-tuning micro-batch (4 x 512 tokens) on an attention projection.
        step("step_int4_m2048", M=2048),
        # The same on an MLP projection at 2 bits.
        step("step_int2_gate_m2048", bits=2, group=64, N=11008, r=16, M=2048),
        # Error correction: rank 32 on a 2-bit projection.
        step("step_int2_r32_m2048", bits=2, group=64, r=32, M=2048),
        # Fine-tuning with dropout on the LoRA branch, a ragged batch.
        step("step_int4_dropout_m1800", M=1800, dropout=0.05),
        # One decoder block of the largest configuration (8 x 512 tokens), forward and backward.
        dict(name="block_int2_m4096", kind="block", bits=2, group=64, hidden=4096, inner=11008, r=8, M=4096, backward=True),
        # The training loss over the vocabulary, 4 x 512 tokens.
        dict(name="loss_t2048_v32000", kind="loss", T=2048, V=32000),
        # Quantizing an MLP weight.
        dict(name="quantize_int4_4096_11008", kind="quantize", bits=4, group=128, K=4096, N=11008),
    ]


def _spread(rng, lo, hi, multiple=1):
    """A size between lo and hi, uniform in its logarithm, rounded to a multiple."""
    return max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / multiple)) * multiple)


def draw(rng):
    kind = rng.choices(("step", "block", "loss", "quantize"), (0.7, 0.12, 0.09, 0.09))[0]
    bits = rng.choice(BITS)
    if kind == "loss":
        return dict(kind=kind, T=_spread(rng, 16, 4096), V=_spread(rng, 4096, 32768, 8))
    if kind == "quantize":
        return dict(kind=kind, bits=bits, group=rng.choice((32, 64, 128)), K=_spread(rng, 512, 8192, 128), N=_spread(rng, 512, 11008, 8))
    if kind == "block":
        hidden, inner = rng.choice(((1024, 2816), (2048, 5632), (4096, 11008)))
        return dict(kind=kind, bits=bits, group=rng.choice((64, 128)), hidden=hidden, inner=inner, r=rng.choice((8, 16, 32)),
                    M=_spread(rng, 1, 16) if rng.random() < 0.5 else _spread(rng, 17, 3072), backward=rng.random() < 0.5)
    K, N = _spread(rng, 512, 8192, 128), _spread(rng, 512, 8192, 64)
    group = rng.choices((32, 64, 128, K), (0.15, 0.35, 0.4, 0.1))[0]
    M = _spread(rng, 1, 8192)
    while M * K * N > 4096 * 4096 * 11008 // (16 if group == 32 else 1):
        M = M // 2 + 1
    option = rng.choices(("", "dropout", "act_order"), (0.6, 0.2, 0.2))[0]
    case = step(None, bits=bits, group=group, K=K, N=N, r=rng.choice((8, 8, 16, 32, 64)), M=M, layers=rng.choice((1, 4)) if M <= 128 else 1,
                backward=rng.random() < 0.75, dropout=0.05 if option == "dropout" else 0.0, act_order=option == "act_order")
    del case["name"]
    return case


class Projection:
    """One quantized projection with its adapter, and the buffers a training program keeps for it."""

    def __init__(self, gen, bits, group, K, N, r, M, backward):
        self.desc = ql.desc(bits, group, K, N, r, 2.0 * r)
        self.K, self.N, self.M = K, N, M
        dev = gen.device
        self.Q = torch.empty((K * bits // 32, N), dtype=torch.int32, device=dev)
        self.scales = torch.empty((K // group, N), dtype=torch.float16, device=dev)
        self.zeros = torch.empty((K // group, N), dtype=torch.float16, device=dev)
        ql.qlora_quantize_rtn(self.desc, torch.randn((N, K), device=dev, generator=gen) * 0.02, self.Q, self.scales, self.zeros)
        self.A = ((torch.rand((r, K), device=dev, generator=gen) * 2 - 1) / math.sqrt(K)).bfloat16()
        self.B = (torch.randn((N, r), device=dev, generator=gen) * 0.01).bfloat16()
        self.Y = torch.empty((M, N), dtype=torch.bfloat16, device=dev)
        self.H = self.G = None
        if backward:
            self.H, self.G = (torch.empty((M, r), dtype=torch.float32, device=dev) for _ in range(2))
            self.dX = torch.empty((M, K), dtype=torch.bfloat16, device=dev)
            self.dA = torch.empty((r, K), dtype=torch.float32, device=dev)
            self.dB = torch.empty((N, r), dtype=torch.float32, device=dev)
            # which pair of backward calls is the cheaper one for this shape, as the library tells
            self.fused_db = ql.qlora_bwd_input_db_on_producers(self.desc, M)

    def forward(self, X, ws):
        self.X = X
        ql.qlora_fwd(self.desc, self.M, X, self.Q, self.scales, self.zeros, self.A, self.B, self.Y, self.H, ws)

    def backward(self, dY, ws):
        if self.fused_db:
            ql.qlora_bwd_input_db(self.desc, self.M, dY, self.Q, self.scales, self.zeros, self.A, self.B, self.H, self.dX, self.G, self.dB, 0, ws)
            ql.qlora_bwd_lora(self.desc, self.M, self.X, None, self.A, self.B, None, self.G, self.dA, None, 0, ws)
        else:
            ql.qlora_bwd_input(self.desc, self.M, dY, self.Q, self.scales, self.zeros, self.A, self.B, self.dX, self.G, ws)
            ql.qlora_bwd_lora(self.desc, self.M, self.X, dY, self.A, self.B, self.H, self.G, self.dA, self.dB, 0, ws)

    def outputs(self):
        return (self.Y,) if self.H is None else (self.Y, self.dX, self.dA, self.dB)


class ActOrderProjection(Projection):
    """A checkpoint quantized in activation order: columns are gathered on the way in and put back on the way out."""

    def __init__(self, gen, bits, group, K, N, r, M, backward):
        super().__init__(gen, bits, group, K, N, r, M, backward)
        perm = torch.randperm(K, device=gen.device, generator=gen)
        self.perm, self.inverse = perm.int(), torch.argsort(perm).int()
        self.A_user, self.X_g, self.A_g = self.A, torch.empty((M, K), dtype=torch.bfloat16, device=gen.device), torch.empty_like(self.A)
        self.A = self.A_g
        if backward:
            self.dX_user, self.dA_user = torch.empty_like(self.dX), torch.empty_like(self.dA)

    def forward(self, X, ws):
        ql.qlora_gather_columns(X, self.perm, self.X_g)
        ql.qlora_gather_columns(self.A_user, self.perm, self.A_g)
        super().forward(self.X_g, ws)

    def backward(self, dY, ws):
        super().backward(dY, ws)
        ql.qlora_gather_columns(self.dX, self.inverse, self.dX_user)
        ql.qlora_gather_columns(self.dA, self.inverse, self.dA_user)

    def outputs(self):
        return (self.Y,) if self.H is None else (self.Y, self.dX_user, self.dA_user, self.dB)


class DropoutProjection(Projection):
    """LoRA dropout: the mask of the step is drawn by the caller."""

    def __init__(self, gen, bits, group, K, N, r, M, backward, dropout):
        super().__init__(gen, bits, group, K, N, r, M, backward)
        self.mask = (torch.rand((M, K), device=gen.device, generator=gen) >= dropout).to(torch.uint8)
        self.keep_scale = 1.0 / (1.0 - dropout)

    def forward(self, X, ws):
        self.X = X
        ql.qlora_fwd_dropout(self.desc, self.M, X, self.mask, self.keep_scale, self.Q, self.scales, self.zeros, self.A, self.B, self.Y, self.H, ws)

    def backward(self, dY, ws):
        ql.qlora_bwd_input_dropout(self.desc, self.M, dY, self.mask, self.keep_scale, self.Q, self.scales, self.zeros, self.A, self.B, self.dX,
                                   self.G, ws)
        ql.qlora_bwd_lora_dropout(self.desc, self.M, self.X, self.mask, self.keep_scale, dY, self.A, self.B, self.H, self.G, self.dA, self.dB, 0, ws)


def _workspace(projections):
    need = max(ql.qlora_workspace_bytes(p.desc, p.M) for p in projections)
    return torch.empty(max(need, 256), dtype=torch.uint8, device=projections[0].Q.device)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def randn(*shape):
        return torch.randn(shape, device="cuda", generator=gen).bfloat16()

    kind = case["kind"]
    if kind == "step":
        args = [case[k] for k in ("bits", "group", "K", "N", "r", "M", "backward")]
        if case["dropout"] > 0.0:
            projections = [DropoutProjection(gen, *args, case["dropout"]) for _ in range(case["layers"])]
        else:
            projections = [(ActOrderProjection if case["act_order"] else Projection)(gen, *args) for _ in range(case["layers"])]
        # the layers' outputs lie behind one another, one tensor for each kind of output
        names = ("Y", "dX_user", "dA_user", "dB") if hasattr(projections[0], "dX_user") else ("Y", "dX", "dA", "dB")
        outputs = []
        for name in names if case["backward"] else names[:1]:
            whole = torch.stack([getattr(p, name) for p in projections])
            for p, part in zip(projections, whole):
                setattr(p, name, part)
            outputs.append(whole)
        return dict(kind=kind, projections=projections, X=[randn(case["M"], case["K"]) for _ in projections],
                    dY=[randn(case["M"], case["N"]) for _ in projections] if case["backward"] else None, outputs=outputs,
                    ws=_workspace(projections))
    if kind == "block":
        width = {1: case["hidden"], 2: case["inner"]}
        P = {name: Projection(gen, case["bits"], case["group"], width[i], width[o], case["r"], case["M"], case["backward"]) for name, i, o in BLOCK}
        state = dict(kind=kind, P=P, x=randn(case["M"], case["hidden"]), ws=_workspace(list(P.values())), backward=case["backward"])
        if case["backward"]:
            state["dY"] = {name: randn(case["M"], P[name].N) for name in ("down", "up", "v", "k")}
        return state
    if kind == "loss":
        T, V = case["T"], case["V"]
        teacher = torch.randn((T, V), device="cuda", generator=gen) * 2.5
        student = (teacher + torch.randn((T, V), device="cuda", generator=gen)).bfloat16()
        return dict(kind=kind, student=student, teacher=teacher.bfloat16(),
                    labels=torch.randint(0, V, (T,), device="cuda", generator=gen).int(), grad_scale=1.0 / T,
                    loss=torch.empty((T,), dtype=torch.float32, device="cuda"), grad=torch.empty_like(student))
    bits, group, K, N = (case[k] for k in ("bits", "group", "K", "N"))
    return dict(kind=kind, desc=ql.desc(bits, group, K, N, 0, 0.0), W=torch.randn((N, K), device="cuda", generator=gen) * 0.02,
                Q=torch.empty((K * bits // 32, N), dtype=torch.int32, device="cuda"),
                scales=torch.empty((K // group, N), dtype=torch.float16, device="cuda"),
                zeros=torch.empty((K // group, N), dtype=torch.float16, device="cuda"))


def run(state):
    kind = state["kind"]
    if kind == "step":
        ws = state["ws"]
        for p, x in zip(state["projections"], state["X"]):
            p.forward(x, ws)
        if state["dY"] is not None:
            for p, dy in zip(reversed(state["projections"]), reversed(state["dY"])):
                p.backward(dy, ws)
        return state["outputs"]
    if kind == "block":
        P, ws, x = state["P"], state["ws"], state["x"]
        source = {"o": "q", "gate": "o", "up": "o", "down": "gate"}
        for name, p in P.items():
            p.forward(P[source[name]].Y if name in source else x, ws)
        if state["backward"]:
            dY = state["dY"]
            below = {"gate": "down", "o": "gate", "q": "o"}
            for name in reversed(P):
                P[name].backward(P[below[name]].dX if name in below else dY[name], ws)
        return {name: p.outputs() for name, p in P.items()}
    if kind == "loss":
        ql.qlora_lrec_loss(state["student"], state["teacher"], state["labels"], 1.0, 0.5, state["grad_scale"], state["loss"], state["grad"])
        return state["loss"], state["grad"]
    ql.qlora_quantize_rtn(state["desc"], state["W"], state["Q"], state["scales"], state["zeros"])
    return state["Q"], state["scales"], state["zeros"]


def _projection_work(bits, group, K, N, r, M, backward, dropout=False):
    weights = K * N * bits / 8 + 4 * (K // group) * N + 2 * r * (K + N)
    forward = weights + 2 * M * (K + N) + (M * K if dropout else 0)
    flops = 2 * M * K * N + 2 * M * r * (K + N)
    if not backward:
        return forward, flops
    return forward + 2 * M * (K + N) + 4 * r * (K + N), 2 * flops + 2 * M * r * (K + N)


def work(case):
    kind = case["kind"]
    if kind == "step":
        b, f = _projection_work(*[case[k] for k in ("bits", "group", "K", "N", "r", "M", "backward")], case["dropout"] > 0.0)
        return {"bytes": b * case["layers"], "flops": f * case["layers"]}
    if kind == "block":
        width = {1: case["hidden"], 2: case["inner"]}
        parts = [_projection_work(case["bits"], case["group"], width[i], width[o], case["r"], case["M"], case["backward"]) for _, i, o in BLOCK]
        return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}
    if kind == "loss":
        n = case["T"] * case["V"]
        return {"bytes": 6 * n + 8 * case["T"], "flops": 16 * n}
    n = case["K"] * case["N"]
    return {"bytes": 4 * n + n * case["bits"] / 8 + 4 * n / case["group"], "flops": 6 * n}


def tolerance(case):
    if case["kind"] == "quantize":
        return "exact"
    # About four times the largest difference seen from the same sums in 64 bits: Y and dX 2.4e-3 (weights, s * H and the
    # output each rounded to bf16 once; 2.8e-3 with dropout, where dX is rounded twice), the loss's gradient 5e-4; largest
    # single difference 1.2e-2 and 3.9e-3.
    if case["kind"] == "loss":
        return {"rel": 2e-3, "max": 1.6e-2}
    if case["kind"] == "step":
        return {"rel": 1e-2, "max": 5e-2}
    # A block's activations pass through four projections and its gradients through four more, each rounded to bf16 (seen:
    # 5.4e-3 and 2.9e-2).
    return {"rel": 2e-2, "max": 1e-1}


# The same results in 64 bits, by plain torch.  Only the inputs come from prepare().

def _weight(p):
    """W [N, K] = scale * (q - zero): 32 consecutive codes of a column are a little-endian bit stream in `bits` words."""
    b, K, N = p.desc.bits, p.K, p.N
    words = (p.Q.long() & 0xFFFFFFFF).reshape(K // 32, b, N)
    codes = torch.empty((K // 32, 32, N), dtype=torch.int64, device=words.device)
    for i in range(32):
        w, off = divmod(i * b, 32)
        q = words[:, w] >> off
        if off + b > 32:
            q = q | (words[:, w + 1] << (32 - off))
        codes[:, i] = q & ((1 << b) - 1)
    groups = p.scales.shape[0]
    W = p.scales.double()[:, None] * (codes.reshape(groups, K // groups, N).double() - p.zeros.double()[:, None])
    return W.reshape(K, N).t()


def _exact_forward(p, X):
    W, s, A, B = _weight(p), p.desc.alpha / p.desc.r if p.desc.r else 0.0, p.A_user if hasattr(p, "A_user") else p.A, p.B
    A, B = A.double(), B.double()
    if hasattr(p, "inverse"):
        W = W[:, p.inverse.long()]
    XD = X * p.mask.double() * p.keep_scale if hasattr(p, "mask") else X
    H = XD @ A.t()
    return X @ W.t() + s * (H @ B.t()), (W, s, A, B, XD, H)


def _exact_backward(p, dY, kept):
    W, s, A, B, XD, H = kept
    G = dY @ B
    low = s * (G @ A)
    if hasattr(p, "mask"):
        low = low * p.mask.double() * p.keep_scale
    return dY @ W + low, s * (G.t() @ XD), s * (dY.t() @ H)


def exact(case, seed):
    kind = case["kind"]
    state = prepare(case, seed)
    if kind == "quantize":
        return None                       # whole numbers and bytes: compared bit by bit
    if kind == "loss":
        logp, logq = (torch.log_softmax(state[k].double(), dim=1) for k in ("student", "teacher"))
        p, labels = logp.exp(), state["labels"].long()[:, None]
        kl = (p * (logp - logq)).sum(dim=1)
        grad = p * (logp - logq - kl[:, None]) + 0.5 * p
        grad.scatter_add_(1, labels, torch.full_like(labels, -0.5, dtype=torch.float64))
        return kl - 0.5 * logp.gather(1, labels)[:, 0], grad * state["grad_scale"]
    if kind == "step":
        out = []
        for i, p in enumerate(state["projections"]):
            Y, kept = _exact_forward(p, state["X"][i].double())
            out.append((Y, *_exact_backward(p, state["dY"][i].double(), kept)) if case["backward"] else (Y,))
        return [torch.stack(parts) for parts in zip(*out)]
    source = {"o": "q", "gate": "o", "up": "o", "down": "gate"}
    below = {"gate": "down", "o": "gate", "q": "o"}
    Y, kept, back = {}, {}, {}
    for name, p in state["P"].items():
        Y[name], kept[name] = _exact_forward(p, Y[source[name]] if name in source else state["x"].double())
    if not case["backward"]:
        return {name: (y,) for name, y in Y.items()}
    for name in reversed(state["P"]):
        dY = back[below[name]][0] if name in below else state["dY"][name].double()
        back[name] = _exact_backward(state["P"][name], dY, kept[name])
    return {name: (Y[name], *back[name]) for name in Y}
