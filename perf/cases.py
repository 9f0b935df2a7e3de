"""The work this library is used for, as timed cases: whole layers and a decoder block through Algorithm 1, calibration
batches into the Hessian, the lazy and the exact variants, and the stored record of a layer.

Shapes are those of the benchmark's configurations (Llama-3-8B-, Llama-3.1-405B- and BERT-base-shaped layers), of the
tests (small, odd and ragged layers), and generic sizes between them.  Inputs are synthetic with the distributions of
the benchmark's recipes: Gaussian weights with outliers, activations that share a low-rank part (ill-conditioned
Hessians, heavy-tailed inverse diagonals) or are products of two Gaussians, with log-normal channel scales."""
import math

import torch

import paper_2407_10032_b200 as lq

_HANDLES = {}


def _handle():
    """One handle per device for the life of the process, as a program that quantises many layers keeps it."""
    dev = torch.cuda.current_device()
    if dev not in _HANDLES:
        _HANDLES[dev] = lq.lq_create(dev)
    return _HANDLES[dev]


# ---------------------------------------------------------------------------------------- cases --
def _layer(name, r, c, n, chunk=0, **kw):
    case = dict(kind="layer", r=r, c=c, n=n, chunk=chunk, dtype="bf16", inputs="low_rank", grid="nonuniform", bits=4, group=0,
                T=2048, t=409, act_order=False)
    case.update(kw)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # a small layer in full precision, the first benchmark configuration: every launch and the serial chain show
        _layer("small-fp32-512", 512, 512, 8192, dtype="fp32", inputs="scaled"),
        # an odd-sized layer quantised in activation order, 3-bit
        _layer("ragged-actorder-1000x1412", 1000, 1412, 5000, bits=3, act_order=True),
        # the attention projection of an 8B model on the paper's calibration set (128 x 2048 tokens): the headline
        _layer("q_proj-4096-nu4", 4096, 4096, 262144),
        # affine grids of 128 weights at the paper's granularity of the search (T = 2048, t = 0.2 T)
        _layer("attn-4096-aff4g128-T2048", 4096, 4096, 65536, inputs="gated", grid="affine", group=128),
        # the MLP down projection of an 8B model: a wide Hessian, 100 candidates per group, calibration in two calls
        _layer("down_proj-14336-aff4g128", 4096, 14336, 131072, chunk=65536, inputs="gated", grid="affine", group=128, T=45, t=9),
        # a whole decoder block of an 8B model in order, 3-bit, with its packed records: seven layers on four Hessians
        dict(name="block-8b-nu3", kind="stack", hidden=4096, kv=1024, mlp=14336, n=131072, bits=3),
        # the tallest layer: the up projection of a 405B model at 2 bits, calibration streamed 8192 tokens at a time
        _layer("up_proj-405b-nu2", 53248, 16384, 65536, chunk=8192, inputs="gated", bits=2),
        # the widest layer that a program holds beside others: 28672 input features, 3-bit
        _layer("wide-28672-nu3", 8192, 28672, 65536, chunk=8192, inputs="gated", bits=3),
        # calibration only: activations as a model produces them (tokens x features), one call per batch of 8 sequences
        dict(name="calib-token-major-4096", kind="calib", c=4096, n=131072, chunk=16384, dtype="bf16"),
        # (S, Z) fitted when the column loop reaches the group, the usual practice of GPTQ implementations
        _layer("lazy-4096-aff4g128", 4096, 4096, 32768, inputs="gated", grid="affine", group=128, T=45, t=9, kind="lazy"),
        # Algorithm 2 on a BERT-base attention layer
        _layer("exact-768-nu4", 768, 768, 16384, kind="exact"),
        # a quantised layer into its stored record and back to bf16 weights
        dict(name="record-14336x4096-nu3", kind="record", r=14336, c=4096, grid="nonuniform", bits=3, group=0),
    ]


def _log_int(rng, lo, hi, step):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step))


def _cost(case):
    """A rough time in ms, to keep drawn cases below the largest listed one."""
    if case["kind"] in ("calib", "record"):
        return 1.0
    r, c, n = case["r"], case["c"], case["n"]
    ms = c * c * n / 1.1e12 + 6e-11 * c ** 3 * 0.25 + c * 0.8e-3 + r * c * c / 1.5e11
    if case["grid"] == "affine":
        ms += r * c * (2.5e-6 if case["T"] == 2048 else 1.5e-7)
    else:
        ms += r * c * 3e-8
    return ms


def draw(rng):
    while True:
        kind = rng.choice(["layer"] * 6 + ["calib", "calib", "lazy", "exact", "record", "stack"])
        if kind == "layer":
            case = _layer(None, _log_int(rng, 96, 53248, 1), _log_int(rng, 256, 16384, 4), _log_int(rng, 2048, 262144, 8),
                          bits=rng.choice([2, 3, 4]), inputs=rng.choice(["low_rank", "gated"]))
            if rng.random() < 0.4:
                g = rng.choice([32, 64, 128, 128, 128, 0])
                T = rng.choice([2048, 45])
                case.update(grid="affine", group=g, T=T, t=int({4: 0.2, 3: 0.3, 2: 0.4}[case["bits"]] * T))
                if g:
                    case["c"] = max(g, case["c"] // g * g)
            if case["c"] <= 4096 and case["n"] <= 32768 and rng.random() < 0.25:
                case.update(dtype="fp32", inputs="scaled")
            if rng.random() < 0.2:
                case["act_order"] = True
            if rng.random() < 0.5:
                case["chunk"] = rng.choice([2048, 8192, 32768])
        elif kind == "calib":
            case = dict(kind="calib", c=_log_int(rng, 512, 14336, 4), n=_log_int(rng, 4096, 131072, 8),
                        chunk=rng.choice([2048, 8192, 16384, 32768]), dtype=rng.choice(["bf16", "bf16", "fp32"]))
            if case["dtype"] == "fp32":
                case["n"] = min(case["n"], 32768)
        elif kind == "lazy":
            g = rng.choice([64, 128, 256])
            case = _layer(None, _log_int(rng, 256, 8192, 1), _log_int(rng, 512, 8192, g), _log_int(rng, 4096, 65536, 8),
                          inputs="gated", grid="affine", group=g, bits=rng.choice([3, 4]), T=45, t=9, kind="lazy")
        elif kind == "exact":
            case = _layer(None, _log_int(rng, 64, 1024, 1), _log_int(rng, 128, 768, 4), _log_int(rng, 2048, 32768, 8),
                          bits=rng.choice([3, 4]), kind="exact")
        elif kind == "record":
            grid = rng.choice(["nonuniform", "affine"])
            case = dict(kind="record", r=_log_int(rng, 256, 16384, 1), c=_log_int(rng, 512, 16384, 128), grid=grid,
                        bits=rng.choice([2, 3, 4]), group=128 if grid == "affine" else 0)
        else:
            case = dict(kind="stack", hidden=_log_int(rng, 512, 4096, 128), kv=_log_int(rng, 128, 1024, 64),
                        mlp=_log_int(rng, 1024, 12288, 128), n=_log_int(rng, 8192, 65536, 8), bits=rng.choice([2, 3, 4]))
            return case
        if "chunk" in case and kind != "calib":
            case["n"] = max(case["n"], 2 * case["c"])       # a calibration set has more tokens than the layer has features
        if _cost(case) <= 200.0:
            return case


# --------------------------------------------------------------------------------------- inputs --
def _gen(seed, k):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + 7919 * k) % (2 ** 63 - 1))
    return g


def _randn(shape, g):
    return torch.randn(shape, generator=g, device="cuda")


def _weights(r, c, seed, k, dtype, outliers):
    g = _gen(seed, k)
    W = _randn((r, c), g) * 0.02
    if outliers == "columns":
        W[:, torch.randperm(c, generator=g, device="cuda")[:4]] *= 10.0
    else:
        W[torch.rand((r, c), generator=g, device="cuda") < 1e-3] *= 20.0
    return W.to(dtype)


def _inputs(c, n, seed, k, dtype, kind, token_major=False):
    g = _gen(seed, 100 + k)
    X = torch.empty((n, c) if token_major else (c, n), device="cuda", dtype=dtype)
    scale = torch.exp((0.5 if kind == "gated" else 1.0) * _randn((c, 1), g))
    rank = {"low_rank": 256, "gated": 64, "scaled": 0}[kind]
    rank = min(rank, max(1, c // 4))
    F = _randn((c, rank), g) / rank ** 0.5
    if kind == "scaled":
        scale[torch.randperm(c, generator=g, device="cuda")[:8]] *= 50.0
    for j in range(0, n, 16384):
        m = min(16384, n - j)
        if kind == "scaled":
            x = _randn((c, m), g)
        elif kind == "low_rank":
            x = F @ _randn((rank, m), g) + 0.05 * _randn((c, m), g)
        else:
            x = (F @ _randn((rank, m), g) + 0.5 * _randn((c, m), g)) * _randn((c, m), g)
        x *= scale
        if token_major:
            X[j:j + m] = x.t()
        else:
            X[:, j:j + m] = x
    return X


def _config(case):
    return lq.Config.make(grid=case["grid"], bits=case["bits"], p=4.0, n_iter=20, group=case["group"], T=case.get("T", 2048),
                          t=case.get("t", 409))


def prepare(case, seed):
    h = _handle()
    kind = case["kind"]
    dtype = torch.float32 if case.get("dtype") == "fp32" else torch.bfloat16
    s = dict(case=case, h=h)
    if kind == "calib":
        c, n, chunk = case["c"], case["n"], min(case["chunk"], case["n"])
        s["X"] = _inputs(c, n, seed, 0, dtype, "low_rank", token_major=True)
        s["H"] = torch.zeros((c, c), device="cuda")
        s["ws"] = torch.empty((max(256, lq.lq_hessian_workspace(dtype, c, chunk, token_major=True)),), device="cuda", dtype=torch.uint8)
    elif kind == "stack":
        hid, kv, mlp, n = case["hidden"], case["kv"], case["mlp"], case["n"]
        groups = [(hid, [hid, kv, kv]), (hid, [hid]), (hid, [mlp, mlp]), (mlp, [hid])]
        cfg = lq.Config.make(grid="nonuniform", bits=case["bits"], p=4.0, n_iter=20)
        s["pass"] = lq.StackPass(h, groups, cfg)
        s["X"] = [_inputs(c, n, seed, g, dtype, "gated" if g == 3 else "low_rank") for g, (c, _) in enumerate(groups)]
        s["W"] = [[_weights(r, c, seed, 10 * g + l, dtype, "entries") for l, r in enumerate(rs)] for g, (c, rs) in enumerate(groups)]
    elif kind == "record":
        r, c = case["r"], case["c"]
        g = _gen(seed, 0)
        s["cfg"] = _config(case)
        s["codes"] = torch.randint(0, 1 << case["bits"], (r, c), generator=g, device="cuda", dtype=torch.uint8)
        s["grid"] = s["scale"] = s["zero"] = None
        if case["grid"] == "nonuniform":
            s["grid"] = (_randn((r, 1 << case["bits"]), g) * 0.03).sort(dim=1).values.contiguous()
        else:
            ng = c // case["group"]
            s["scale"] = 0.004 + 0.002 * torch.rand((r, ng), generator=g, device="cuda")
            s["zero"] = torch.randint(0, 1 << case["bits"], (r, ng), generator=g, device="cuda", dtype=torch.int32)
        s["record"] = torch.zeros((lq.lq_pack_layer_bytes(s["cfg"], r, c)[0],), device="cuda", dtype=torch.uint8)
        s["W_hat"] = torch.empty((r, c), device="cuda", dtype=torch.bfloat16)
    else:
        r, c, n = case["r"], case["c"], case["n"]
        s["chunk"] = min(case["chunk"], n) or n
        s["cfg"] = cfg = _config(case)
        s["W"] = _weights(r, c, seed, 0, dtype, "columns" if case["inputs"] == "scaled" else "entries")
        s["X"] = _inputs(c, n, seed, 0, dtype, case["inputs"])
        P = s["pass"] = lq.LayerPass(h, r, c, cfg, w_dtype=dtype, x_dtype=dtype, n_chunk=s["chunk"], want_w_hat=False,
                                     act_order=case["act_order"])
        need = {"layer": 0, "lazy": lq.lq_quantize_layer_lazy_workspace, "exact": lq.lq_quantize_exact_workspace}[kind]
        if need:
            s["ws"] = torch.empty((max(need(cfg, r, c), P.ws.numel()),), device="cuda", dtype=torch.uint8)
    return s


# ------------------------------------------------------------------------------------- one pass --
def run(s):
    case, h = s["case"], s["h"]
    kind = case["kind"]
    if kind == "calib":
        s["H"].zero_()
        for j in range(0, case["n"], case["chunk"]):
            lq.lq_hessian_accumulate(h, s["X"][j:j + case["chunk"]], s["H"], 2.0, s["ws"], token_major=True)
        lq.lq_hessian_finalize(h, s["H"])
        return s["H"]
    if kind == "stack":
        S = s["pass"]
        S.run(s["X"], s["W"])
        return [[dict(codes=P.codes, grid=P.grid, loss=P.loss) for P in ps] for ps in S.passes]
    if kind == "record":
        lq.lq_pack_layer(h, s["cfg"], s["codes"], s["grid"], s["scale"], s["zero"], s["record"])
        lq.lq_unpack_layer(h, s["cfg"], s["record"], case["r"], case["c"], s["W_hat"])
        return s["record"], s["W_hat"]
    P, W, X, chunk = s["pass"], s["W"], s["X"], s["chunk"]
    if kind == "layer" and chunk == case["n"]:
        P.run(W, X)
    else:
        P.H.zero_()
        for j in range(0, case["n"], chunk):
            P.accumulate(X[:, j:j + chunk])
        if kind == "layer":
            P.finish(W)
        else:
            lq.lq_hessian_finalize(h, P.H)
            lq.lq_prepare_hinv(h, P.H, P.U, P.dinv, P.ws, 0.01, W)
            if kind == "lazy":
                lq.lq_quantize_layer_lazy(h, s["cfg"], W, P.U, P.dinv, P.scale, P.zero, P.codes, s["ws"], P.W_hat, P.loss)
            else:
                lq.lq_fit_grid(h, s["cfg"], W, P.dinv, P.ws, P.grid, P.scale, P.zero)
                lq.lq_quantize_exact(h, s["cfg"], W, P.U, P.codes, s["ws"], P.grid, P.scale, P.zero, P.W_hat, P.loss)
    out = dict(codes=P.codes, loss=P.loss, dinv=P.dinv)
    if P.grid is not None:
        out["grid"] = P.grid
    else:
        out["scale"], out["zero"] = P.scale, P.zero
    return out


# ------------------------------------------------------------------------------------ in 64 bits --
def exact(case, seed):
    """H and diag((H + damp I)^-1) in 64 bits.  Codes, grids and losses have no entry: a weight within fp32 rounding of a
    midpoint goes either way and takes the rest of its row along, so what they are off by is luck and not precision (the
    tolerance below bounds it); an activation-ordered layer has its dinv in an order that rounding of H decides."""
    kind, c, n = case["kind"], case.get("c", 0), case.get("n", 0)
    if kind in ("stack", "record") or c > 16384 or case.get("act_order"):
        return None
    dtype = torch.float32 if case.get("dtype") == "fp32" else torch.bfloat16
    X = _inputs(c, n, seed, 0, dtype, "low_rank" if kind == "calib" else case["inputs"], token_major=kind == "calib")
    H = torch.zeros((c, c), device="cuda", dtype=torch.float64)
    for j in range(0, n, 16384):
        x = X[j:j + 16384].t().double() if kind == "calib" else X[:, j:j + 16384].double()
        H.addmm_(x, x.t(), alpha=2.0)
    if kind == "calib":
        return H
    H.diagonal().add_(0.01 * H.diagonal().mean())
    R_inv = torch.linalg.solve_triangular(torch.linalg.cholesky(H), torch.eye(c, device="cuda", dtype=torch.float64), upper=False)
    out = dict(codes=None, loss=None, dinv=R_inv.square_().sum(dim=0))
    out.update(dict(grid=None) if case["grid"] == "nonuniform" else dict(scale=None, zero=None))
    return out


# ------------------------------------------------------------------------------- floors, limits --
def _layer_work(r, c, n, elem, K, exact=False):
    """X and W read, codes and tables written; X X^T by symmetry, the factor of the inverse, the column loop's updates."""
    nbytes = elem * (c * n + r * c) + r * c + 4 * r * K
    flops = c * c * n + 2 * c ** 3 / 3 + (2 * r * c ** 3 / 6 if exact else r * c * c)
    return nbytes, flops


def work(case):
    kind = case["kind"]
    if kind == "calib":
        elem = 4 if case["dtype"] == "fp32" else 2
        return {"bytes": elem * case["c"] * case["n"] + 4 * case["c"] ** 2, "flops": case["c"] ** 2 * case["n"]}
    if kind == "record":
        rc = case["r"] * case["c"]
        return {"bytes": rc + 2 * rc * case["bits"] / 8 + 2 * rc, "flops": rc}
    if kind == "stack":
        hid, kv, mlp, n, K = case["hidden"], case["kv"], case["mlp"], case["n"], 1 << case["bits"]
        nbytes = flops = 0
        for c, rs in [(hid, [hid, kv, kv]), (hid, [hid]), (hid, [mlp, mlp]), (mlp, [hid])]:
            b, f = _layer_work(sum(rs), c, n, 2, K)
            nbytes, flops = nbytes + b, flops + f
        return {"bytes": nbytes, "flops": flops}
    nbytes, flops = _layer_work(case["r"], case["c"], case["n"], 4 if case["dtype"] == "fp32" else 2,
                                (1 << case["bits"]) if case["grid"] == "nonuniform" else 2 * case["c"] // (case["group"] or case["c"]),
                                kind == "exact")
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Four times what the same pass gives with its tokens in another order (fp32 sums in another order), which is what
    the fp32 Hessian and working copy of the weights leave open: a near-tie that falls the other way changes the codes of
    the rest of its row.  Seen that way: codes 1.4e-3 apart (non-uniform grids on ill-conditioned Hessians), 1.2e-4
    (affine), 1.0e-3 (Algorithm 2); layer loss 5e-4; scales 2.5e-3 where one group took the other of two candidates; one
    centroid of a whole layer 0.25 of the grids' root mean square away; H 1.7e-7."""
    kind = case["kind"]
    if kind == "record":
        return "exact"
    if kind == "calib":
        return {"rel": 7e-7, "max": 1e-5}
    if case.get("grid") == "affine":
        return {"rel": 1e-2, "max": 0.99, "differ": 1e-3}
    return {"rel": 4e-3, "max": 0.99, "differ": 6e-3}
