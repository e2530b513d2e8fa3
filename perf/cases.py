"""Performance cases of the SubZero+ weight path: what users of the library have it do,
over the sizes, ranks, dtypes and directions it is used with.

Five kinds of work, each through the public entry points (``SubZeroPlus`` and the binding):

* ``step``    -- one whole step of Alg. 3 (``run_step``): the perturbation passes, a loss
  after each (given here: the forward passes are the caller's), and the estimator, Adam
  update and fused restore.  This is what a training run repeats.
* ``refresh`` -- new Haar bases for every matrix (Alg. 1), once every F steps.
* ``linear``  -- one loss evaluation's linear layers at the perturbed weights without a
  weight pass (``linear_prepare``, then ``linear_perturbed`` per matrix), from a few tokens
  to a full batch.
* ``mezo``    -- one full-space step of Eq. (1): +eps, -2 eps, restore fused with the update.
* ``noalloc`` -- one perturbation pass of one matrix without a context.

A case is a dict of plain values.  ``shapes`` lists one layer's matrices as
"m x n [* count], ..."; ``layers`` repeats it.  Values are those the path meets: weights
N(0, 0.02^2), losses 2.0 + 0.01 N(0, 1), moments of a run under way.
"""

import math

import numpy as np
import torch

from paper_2608_15665_gb300 import binding as zb
from paper_2608_15665_gb300.schedule import SubZeroPlus, step_plan

DEVICE = "cuda"
EPS, BETA1, BETA2, EPS_ADAM = 1e-3, 0.9, 0.95, 1e-8
LR = 1e-3
MEZO_LR = 1e-6
START_T = 10          # steps already taken: Adam's bias corrections are those of step 11
REFRESH = 3           # refresh index of the bases in hand

OPT13_LAYER = "2048x2048*4,8192x2048,2048x8192"
LLAMA7_LAYER = "4096x4096*4,11008x4096*2,4096x11008"
DENSE32_LAYER = "8192x5120,1024x5120*2,5120x8192,25600x5120*2,5120x25600"
LORA13_LAYER = "8x5120,5120x8,8x5120,5120x8"


# ---------------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest training set of the repository: one fp32 matrix, a chain of launches
        # of a few microseconds each, where latency and the host path count
        dict(name="step 256x256 f32 r8", kind="step", shapes="256x256", layers=1, dtype="f32",
             r=8, q=4, scheme="central", gamma=False),
        # LoRA fine-tuning of a 13B model: 160 thin fp32 factors that stay in L2; the
        # per-layer gradient norms are logged
        dict(name="step LoRA 13B f32 r4", kind="step", shapes=LORA13_LAYER, layers=40,
             dtype="f32", r=4, q=8, scheme="central", gamma=True),
        # full fine-tuning of a 1.3B model at a small rank
        dict(name="step 1.3B bf16 r16", kind="step", shapes=OPT13_LAYER, layers=24, dtype="bf16",
             r=16, q=4, scheme="central", gamma=False),
        # full fine-tuning of a 7B model, forward differences: the flagship size, every
        # matrix of the model in one pass
        dict(name="step 7B bf16 r32", kind="step", shapes=LLAMA7_LAYER, layers=32, dtype="bf16",
             r=32, q=4, scheme="forward", gamma=False),
        # one pipeline stage (8 of 64 layers) of a 32B model with grouped-query projections
        dict(name="step 32B/8 bf16 r64", kind="step", shapes=DENSE32_LAYER, layers=8,
             dtype="bf16", r=64, q=8, scheme="central", gamma=False),
        # the paper's own scale (rank 128, 99 queries) on one stage (4 of 32 layers) of 7B
        dict(name="step 7B/8 bf16 r128 q99", kind="step", shapes=LLAMA7_LAYER, layers=4,
             dtype="bf16", r=128, q=99, scheme="forward", gamma=False),
        # a small model kept in fp32 (hidden size 768, 12 layers) at an ordinary rank
        dict(name="step 768x12 f32 r32", kind="step", shapes="768x768*4,3072x768,768x3072",
             layers=12, dtype="f32", r=32, q=2, scheme="central", gamma=False),
        # the refresh of a quarter of the 32B model, which runs every 5 steps there
        dict(name="refresh 32B/4 r64", kind="refresh", shapes=DENSE32_LAYER, layers=16,
             dtype="bf16", r=64),
        # the refresh of the LoRA set: many small panels at a small rank
        dict(name="refresh LoRA 13B r4", kind="refresh", shapes=LORA13_LAYER, layers=40,
             dtype="f32", r=4),
        # the linear layers of one 7B block at the perturbed weights, a full batch
        dict(name="linear 7B 4096 tok r32", kind="linear", shapes=LLAMA7_LAYER, layers=1,
             tokens=4096, r=32),
        # the same block on one short example (an odd number of tokens), where reading the
        # weights is what there is to do
        dict(name="linear 7B 97 tok r32", kind="linear", shapes=LLAMA7_LAYER, layers=1,
             tokens=97, r=32),
        # MeZO on the 1.3B set: every weight draws its own Gaussian, three times a step
        dict(name="mezo 1.3B bf16", kind="mezo", shapes=OPT13_LAYER, layers=24, dtype="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _set_of(rng, size_lo, size_hi, step, most_params):
    """Shapes text and layer count of a random set: 1-3 shapes, sizes spread over their
    logarithm in multiples of `step`, at most most_params weights."""
    shapes = []
    for _ in range(rng.randint(1, 3)):
        m = max(size_lo, _log_int(rng, size_lo, size_hi) // step * step)
        n = max(size_lo, _log_int(rng, size_lo, size_hi) // step * step)
        shapes.append((m, n, rng.choice([1, 1, 2, 4])))
    per_layer = sum(m * n * c for m, n, c in shapes)
    layers = max(1, min(_log_int(rng, 1, 32), most_params // per_layer))
    return ",".join(f"{m}x{n}*{c}" for m, n, c in shapes), layers


def draw(rng):
    """One more case of the listed kinds; no dearer than the 7B step."""
    kind = rng.choice(["step"] * 5 + ["refresh"] * 2 + ["linear"] * 2 + ["mezo", "noalloc"])
    if kind == "step":
        family = rng.choice(["small", "lora", "tensor", "tensor", "odd"])
        scheme, gamma = rng.choice(["central", "forward"]), rng.random() < 0.5
        if family == "small":          # small ranks: fp32 or bf16, any width
            shapes, layers = _set_of(rng, 64, 4096, 1, 100_000_000)
            return dict(kind=kind, shapes=shapes, layers=layers, dtype=rng.choice(["f32", "bf16"]),
                        r=rng.choice([4, 8]), q=_log_int(rng, 1, 16), scheme=scheme, gamma=gamma)
        if family == "lora":           # the thin factors of adapters of rank 8 or 16
            a, h = rng.choice([8, 16]), _log_int(rng, 512, 8192)
            return dict(kind=kind, shapes=f"{a}x{h}*2,{h}x{a}*2", layers=_log_int(rng, 4, 80),
                        dtype=rng.choice(["f32", "bf16"]), r=rng.choice([4, 8]),
                        q=_log_int(rng, 2, 16), scheme=scheme, gamma=gamma)
        if family == "tensor":         # bf16, widths a multiple of 8
            r = rng.choice([16, 32, 64, 128])
            shapes, layers = _set_of(rng, 256, 12288, 8, 1_500_000_000)
            return dict(kind=kind, shapes=shapes, layers=layers, dtype="bf16", r=r,
                        q=_log_int(rng, 1, 8), scheme=scheme, gamma=gamma)
        r = rng.choice([16, 32, 64])   # fp32, or bf16 with odd widths, at ordinary ranks
        shapes, layers = _set_of(rng, 129, 3000, 1, 60_000_000)
        return dict(kind=kind, shapes=shapes, layers=layers, dtype=rng.choice(["f32", "bf16"]), r=r,
                    q=_log_int(rng, 1, 4), scheme=scheme, gamma=gamma)
    if kind == "refresh":
        r = rng.choice([4, 8, 16, 32, 64, 128])
        shapes, layers = _set_of(rng, max(64, r), 16384, 8, 1_500_000_000)
        return dict(kind=kind, shapes=shapes, layers=layers, dtype="bf16", r=r)
    if kind == "linear":
        r = rng.choice([16, 32, 64, 128])
        shapes, _ = _set_of(rng, 512, 12288, 8, 400_000_000)
        return dict(kind=kind, shapes=shapes, layers=1, tokens=_log_int(rng, 1, 8192), r=r)
    if kind == "mezo":
        shapes, layers = _set_of(rng, 128, 8192, 1, 500_000_000)
        return dict(kind=kind, shapes=shapes, layers=layers, dtype=rng.choice(["f32", "bf16"]))
    r = rng.choice([4, 8, 16, 32, 64])
    return dict(kind="noalloc", shapes=f"{_log_int(rng, 128, 8192)}x{_log_int(rng, 128, 16384)}",
                layers=1, dtype=rng.choice(["f32", "bf16"]), r=r)


# ---------------------------------------------------------------------------- inputs

def _shapes(case):
    one = []
    for part in case["shapes"].split(","):
        dims, _, count = part.partition("*")
        m, n = dims.split("x")
        one += [(int(m), int(n))] * int(count or 1)
    return one * case["layers"]


def _dtype(case):
    return torch.float32 if case.get("dtype") == "f32" else torch.bfloat16


def _views(sizes, dtype, fill=None):
    """One flat buffer and a view per (rows, cols) of it; rows are padded to a multiple of
    16 bytes, as the library asks for."""
    per = 16 // torch.empty(0, dtype=dtype).element_size()
    padded = [(m, n, -(-n // per) * per) for m, n in sizes]
    flat = torch.zeros(sum(m * ld for m, _, ld in padded), dtype=dtype, device=DEVICE)
    views, at = [], 0
    for m, n, ld in padded:
        views.append(flat[at:at + m * ld].view(m, ld)[:, :n])
        at += m * ld
    return flat, views


def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(seed)


def _weights(case, seed):
    flat, views = _views(_shapes(case), _dtype(case))
    g = _generator(seed)
    for v in views:
        v.copy_(torch.randn(v.shape, generator=g, device=DEVICE).mul_(0.02))
    return flat, views


def _moments(case, seed):
    """M and Vm of a run under way: the scale of G, Vm above M^2's mean."""
    r, q = case["r"], case["q"]
    scale = 7.0 / math.sqrt(q)
    g = _generator(seed + 1)
    k = len(_shapes(case))
    M = torch.randn(k, r, r, generator=g, device=DEVICE).mul_(0.3 * scale)
    Vm = torch.rand(k, r, r, generator=g, device=DEVICE).add_(0.5).mul_(scale * scale)
    return M, Vm


def _losses(case, seed):
    n = {"central": 2 * case["q"], "forward": case["q"] + 1}[case["scheme"]]
    g = np.random.default_rng(seed + 2)
    return (2.0 + 0.01 * g.standard_normal(n)).astype(np.float32)


def _tokens(case, seed):
    """The inputs of the layers: one bf16 matrix per width."""
    g = _generator(seed + 3)
    return {n: torch.randn(case["tokens"], n, generator=g, device=DEVICE).to(torch.bfloat16)
            for n in sorted({n for _, n in _shapes(case)})}


def _mezo_coefs(seed):
    rho = float(np.random.default_rng(seed + 4).standard_normal()) * 7.0
    return [EPS, -2.0 * EPS, EPS - MEZO_LR * rho]


class Bound(SubZeroPlus):
    """SubZeroPlus over flat storage: the weights, bases and moments of all matrices are
    views of one buffer each, as a training program that checkpoints them holds them."""

    def __init__(self, weights, r, q, seed, moments=None):
        self.weights = list(weights)
        self.r, self.q, self.seed = r, q, seed
        self.u_flat, self.U = _views([(W.shape[0], r) for W in weights], torch.float32)
        self.v_flat, self.V = _views([(W.shape[1], r) for W in weights], torch.float32)
        if moments is None:
            moments = [torch.zeros(len(self.weights), r, r, device=DEVICE) for _ in range(2)]
        self.M, self.Vm = moments
        mats = [zb.make_matrix(W, U, V, M, Vm)
                for W, U, V, M, Vm in zip(self.weights, self.U, self.V, self.M, self.Vm)]
        self.stream = None
        self.ctx = zb.zo_create(mats, r, q, seed, 0, None)


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, s.kind, s.t = case, case["kind"], START_T
    if s.kind == "noalloc":
        s.flat, (s.W,) = _weights(case, seed)
        z = Bound([s.W], case["r"], 1, seed)
        z.refresh(REFRESH)
        z.sync()
        s.U, s.V = z.U[0].clone(), z.V[0].clone()
        z.close()
        s.seed = seed
        return s
    if s.kind == "refresh":
        s.flat, views = _views(_shapes(case), _dtype(case))
    else:
        s.flat, views = _weights(case, seed)
    if s.kind == "mezo":
        # the full-space pass needs no bases; the context is bound at the smallest rank
        s.z = Bound(views, 4, 1, seed)
        s.coefs = _mezo_coefs(seed)
        return s
    if s.kind == "step":
        s.z = Bound(views, case["r"], case["q"], seed, _moments(case, seed))
        s.losses = [float(x) for x in _losses(case, seed)]
        s.gamma = (torch.zeros(len(views), device=DEVICE) if case["gamma"] else None)
        s.loss_fn = lambda t, i: s.losses[i]
    else:
        s.z = Bound(views, case["r"], 2, seed)
    s.j = REFRESH
    if s.kind == "linear":
        tokens = _tokens(case, seed)
        s.X = [tokens[n] for _, n in _shapes(case)]
    if s.kind != "refresh":
        s.z.refresh(REFRESH)
    return s


# ---------------------------------------------------------------------------- a pass

def run(s):
    t = s.t
    s.t += 1
    if s.kind == "step":
        c = s.case
        s.z.run_step(t, t + 1, s.loss_fn, c["scheme"], EPS, LR, BETA1, BETA2, EPS_ADAM,
                     gamma_out=s.gamma)
        out = [s.flat, s.z.M, s.z.Vm]
        return out + [s.gamma] if s.gamma is not None else out
    if s.kind == "refresh":
        s.z.refresh(s.j)
        s.j += 1
        return [s.z.u_flat, s.z.v_flat]
    if s.kind == "linear":
        s.z.linear_prepare(t, 1, 1.0, -1, 0.0, EPS)
        return [s.z.linear_perturbed(i, X) for i, X in enumerate(s.X)]
    if s.kind == "mezo":
        for coef in s.coefs:
            s.z.mezo_perturb(t, coef)
        return [s.flat]
    zb.zo_perturb_noalloc(s.W, s.U, s.V, s.case["r"], s.seed, 0, t, 0, 1.0, -1, 0.0, EPS)
    return [s.flat]


def _passes(case):
    return len(step_plan(case["scheme"], case["q"])[0]) + 1


def work(case):
    shapes, r = _shapes(case), case.get("r", 0)
    es = 4 if case.get("dtype") == "f32" else 2
    params = sum(m * n for m, n in shapes)
    panel_rows = sum(m + n for m, n in shapes)
    kind = case["kind"]
    if kind == "step":
        # every pass reads and writes W (a loss is evaluated on each state of it) and
        # needs U and V; the update reads and writes the moments
        p = _passes(case)
        return {"bytes": p * (2 * es * params + 4 * r * panel_rows) + 16 * r * r * len(shapes),
                "flops": p * 2 * r * params}
    if kind == "refresh":
        return {"bytes": 4 * r * panel_rows, "flops": 4 * r * r * panel_rows}
    if kind == "linear":
        T = case["tokens"]
        x = sum({n: T * n for _, n in shapes}.values())
        y = sum(T * m for m, _ in shapes)
        return {"bytes": 2 * (params + x + y) + 4 * r * panel_rows,
                "flops": 2 * T * params + 2 * T * r * panel_rows}
    if kind == "mezo":
        return {"bytes": 3 * 2 * es * params, "flops": 3 * 2 * params}
    return {"bytes": 2 * es * params + 4 * r * panel_rows, "flops": 2 * r * params}


def tolerance(case):
    """About four times what the path shows against itself with its sums in another order
    (the FMA pass against the tensor cores, one GEMM tiling family against the other), or,
    where both orders give the same bits, against 64 bits.

    bf16 results differ by the few elements whose exact value lies at a rounding boundary,
    one unit (2^-8 to 2^-7 of the value) a pass: seen up to rel 1.4e-6, max 0.01 over 17
    passes and rel 1.3e-5, max 0.034 over 100; a bf16 layer rel 7.6e-6, max 7.4e-3.  fp32
    results: rel 2.6e-7, max 8e-7 (5e-6 for a basis); the basis of a nearly square panel,
    whose last columns are ill-conditioned: rel 1.1e-6, max 1.8e-5 (Householder in fp32)."""
    kind = case["kind"]
    if kind == "refresh":
        square = any(min(m, n) < 2 * case["r"] for m, n in _shapes(case))
        return {"rel": 5e-6, "max": 1e-4} if square else {"rel": 1e-6, "max": 2e-5}
    if kind == "linear":
        return {"rel": 3e-5, "max": 0.03}
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 5e-6}
    if kind == "step" and _passes(case) > 40:
        return {"rel": 5e-5, "max": 0.13}
    return {"rel": 1e-5, "max": 0.04}


# ---------------------------------------------------------------------------- 64 bits

M32 = 0xFFFFFFFF


def _mul_hi_lo(a, x):
    """High and low words of a * x for a 32-bit constant a and int64 tensors x < 2^32."""
    hi = (a * (x >> 16) + ((a * (x & 0xFFFF)) >> 16)) >> 16
    return hi, (a * x) & M32


def _normals(seed, x1, x2, x3, c):
    """Box-Muller normals (fp64, four per counter word) of the Philox4x32-10 stream at the
    counter words c (int64; x1, x2, x3 numbers or int64 tensors of c's shape)."""
    full = lambda v: torch.as_tensor(v, dtype=torch.int64, device=DEVICE).expand(c.shape)  # noqa: E731
    w = [c, full(x1), full(x2), full(x3)]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        ha, la = _mul_hi_lo(0xD2511F53, w[0])
        hb, lb = _mul_hi_lo(0xCD9E8D57, w[2])
        w = [hb ^ w[1] ^ k0, lb, ha ^ w[3] ^ k1, la]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    u = [((x >> 8) + 1).double() * 2.0 ** -24 for x in w]
    out = []
    for a, b in ((0, 1), (2, 3)):
        rad = torch.sqrt(-2.0 * torch.log(u[a]))
        out += [rad * torch.cos(2.0 * math.pi * u[b]), rad * torch.sin(2.0 * math.pi * u[b])]
    return torch.stack(out, -1)


def _block(seed, x1, x2, x3, n):
    c = torch.arange((n + 3) // 4, dtype=torch.int64, device=DEVICE)
    return _normals(seed, x1, x2, x3, c).reshape(-1)[:n]


def _z(seed, i, t, k, r):
    return _block(seed, i, t, (1 << 24) | k, r * r).view(r, r)


def _haar(seed, i, j, tag, rows, r):
    omega = _block(seed, i, j, tag << 24, rows * r).view(rows, r)
    Q, R = torch.linalg.qr(omega)
    return Q * torch.where(torch.diagonal(R) < 0, -1.0, 1.0)


def _bases(case, seed, i, j):
    m, n = _shapes(case)[i]
    return _haar(seed, i, j, 2, m, case["r"]), _haar(seed, i, j, 3, n, case["r"])


def _f32(x):
    return float(np.float32(x))


def exact(case, seed):
    kind, shapes, r = case["kind"], _shapes(case), case.get("r")
    if kind == "refresh":
        flats = [[], []]
        for i in range(len(shapes)):
            for f, Q in zip(flats, _bases(case, seed, i, REFRESH)):
                f.append(Q.reshape(-1))
        return [torch.cat(f) for f in flats]
    W0 = _weights(case, seed)[1]
    eps = _f32(EPS)
    if kind == "linear":
        X = _tokens(case, seed)
        out = []
        for i, (m, n) in enumerate(shapes):
            U, V = _bases(case, seed, i, REFRESH)
            C = eps * _z(seed, i, START_T, 1, r)
            out.append(X[n].double() @ (W0[i].double() + U @ (C @ V.T)).T)
        return out
    # the weights, laid out as run() returns them
    per = 16 // W0[0].element_size()
    flat = torch.zeros(sum(m * (-(-n // per) * per) for m, n in shapes), dtype=torch.float64,
                       device=DEVICE)
    at, M_out, V_out, gamma = 0, [], [], []
    if kind == "step":
        q, L = case["q"], torch.from_numpy(_losses(case, seed)).double().to(DEVICE)
        rho = (L[0::2] - L[1::2]) / (2 * eps) if case["scheme"] == "central" else (L[1:] - L[0]) / eps
        M0, Vm0 = _moments(case, seed)
        b1, b2, t1 = _f32(BETA1), _f32(BETA2), START_T + 1
    for i, (m, n) in enumerate(shapes):
        ld = -(-n // per) * per
        W = flat[at:at + m * ld].view(m, ld)[:, :n]
        at += m * ld
        W.copy_(W0[i])
        if kind == "mezo":
            coef = sum(_f32(c) for c in _mezo_coefs(seed))
            n4 = (n + 3) // 4
            rows = max(1, (1 << 25) // n)
            for r0 in range(0, m, rows):
                k = min(rows, m - r0)
                c = torch.arange(r0 * n4, (r0 + k) * n4, dtype=torch.int64, device=DEVICE)
                W[r0:r0 + k] += coef * _normals(seed, i, START_T, 5 << 24, c).view(k, 4 * n4)[:, :n]
            continue
        U, V = _bases(case, seed, i, REFRESH)
        if kind == "noalloc":
            C = eps * _z(seed, i, START_T, 0, r)
        else:
            # the perturbations cancel; what is left is the update
            words = r * r // 4
            k = torch.arange(q, dtype=torch.int64, device=DEVICE).repeat_interleave(words)
            c = torch.arange(words, dtype=torch.int64, device=DEVICE).repeat(q)
            Z = _normals(seed, i, START_T, (1 << 24) | k, c).view(q, r, r)
            G = (rho.view(q, 1, 1) * Z).sum(0) / q
            M = b1 * M0[i].double() + (1 - b1) * G
            Vm = b2 * Vm0[i].double() + (1 - b2) * G * G
            M_out.append(M)
            V_out.append(Vm)
            gamma.append(G.norm())
            C = -_f32(LR) * (M / (1 - b1 ** t1)) / (torch.sqrt(Vm / (1 - b2 ** t1)) + _f32(EPS_ADAM))
        W += U @ (C @ V.T)
    if kind != "step":
        return [flat]
    out = [flat, torch.stack(M_out), torch.stack(V_out)]
    return out + [torch.stack(gamma)] if case["gamma"] else out
