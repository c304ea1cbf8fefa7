"""The workloads whose speed is measured: what a program built on this library has it do.

A case is a plain dict. Its "kind" names the call:

  pipeline  build a handle from labelled samples, solve for the t dominant pairs, project a held-out set: what a
            recognition program runs once per training split
  build     build a handle and read every result of the build back (factors, Grams, K(alpha), eigenvalues)
  apply     one product with exp(alpha S_W), exp(alpha S_B), M or N on a block of b vectors, on a handle in hand: the
            step of a Krylov method that a program writes itself
  solve     block Lanczos on a handle in hand (another t or tolerance on the same training set)
  arnoldi   block Arnoldi, the nonsymmetric form, on a handle in hand
  direct    the exact solve in span[H_W H_B], the library's cross-check of the Krylov solvers
  batched   many independent problems of uneven size at once (random training splits, class subsets)

Samples are drawn as in ``paper_1512_06500_gb300/synth.py`` (class means N(0, 1) per pixel, samples mean + N(0, 0.3^2),
clipped to [0, 1], labels shuffled), on the GPU and from the seed alone. The block sizes, scales tau and sample counts are
those of its workloads. Class sizes run from nj_lo to nj_hi.
"""
import math
import random

import torch

from paper_1512_06500_gb300 import eda

PREC = {"f64": 0, "f32": 1, "bf16": 2, "f64_tc": 4}
OPS = {"SW": 0, "SB": 1, "M": 2, "N": 3}


def listed():
    return [
        # 16 x 16 images, 8 classes: the smallest training set, one call of everything; launches and latency count
        dict(name="pipeline_d256_k8", kind="pipeline", prec="f64", d=256, k=8, nj_lo=6, nj_hi=6, b=1, tau=10.0, t=7,
             tol=1e-10, test=5, x="f64"),
        # 64 x 64 images, 40 people, 5 images each: an ordinary face set, plain FP64
        dict(name="pipeline_d4096_k40", kind="pipeline", prec="f64", d=4096, k=40, nj_lo=5, nj_hi=5, b=8, tau=10.0,
             t=39, tol=1e-10, test=5, x="f64"),
        # 256 x 256 images, 200 people, 10 images each: the largest training set, FP64-accurate tensor-core products
        dict(name="pipeline_d65536_k200_tc", kind="pipeline", prec="f64_tc", d=65536, k=200, nj_lo=10, nj_hi=10, b=32,
             tau=10.0, t=199, tol=1e-6, test=3, x="f64"),
        # 128 x 128 images held in single precision, uneven classes, not tuned for: the whole build result is read,
        # the Grams' eigenvalues among it
        dict(name="build_d16384_k100", kind="build", prec="f64", d=16384, k=100, nj_lo=6, nj_hi=8, b=16, tau=10.0,
             x="f32"),
        # one exp(alpha S_W) product of an ordinary face set in FP64: a few microseconds of work
        dict(name="apply_sw_d4096_k40", kind="apply", prec="f64", op="SW", d=4096, k=40, nj_lo=5, nj_hi=5, b=8,
             tau=10.0),
        # one M product of the largest set with the tensor-core FP64 products: the step of its Krylov iteration
        dict(name="apply_m_d65536_k200_tc", kind="apply", prec="f64_tc", op="M", d=65536, k=200, nj_lo=10, nj_hi=10,
             b=32, tau=10.0),
        # bf16 sweeps: a factor that stays resident in shared memory, and one that streams from HBM
        dict(name="apply_sw_d16384_k100_bf16", kind="apply", prec="bf16", op="SW", d=16384, k=100, nj_lo=7, nj_hi=7,
             b=16, tau=20.0),
        dict(name="apply_sw_d65536_k200_bf16", kind="apply", prec="bf16", op="SW", d=65536, k=200, nj_lo=10, nj_hi=10,
             b=32, tau=20.0),
        # the Krylov solvers alone on 128 x 128 images, 100 people, 7 images each: Lanczos with the tensor-core
        # products, Arnoldi in plain FP64
        dict(name="solve_d16384_k100_tc", kind="solve", prec="f64_tc", d=16384, k=100, nj_lo=7, nj_hi=7, b=16,
             tau=10.0, t=99, tol=1e-6),
        dict(name="arnoldi_d16384_k100", kind="arnoldi", prec="f64", d=16384, k=100, nj_lo=7, nj_hi=7, b=16, tau=10.0,
             t=99, tol=1e-6),
        # the exact solve of the same set size, a ragged image size and uneven classes
        dict(name="direct_d10305_k93_tc", kind="direct", prec="f64_tc", d=10305, k=93, nj_lo=5, nj_hi=9, b=16,
             tau=10.0, t=92),
        # 32 problems of uneven d, k and class sizes at once
        dict(name="batched32", kind="batched", prec="f64", count=32, shapes=5000, d_lo=1024, d_hi=16384, k_lo=10,
             k_hi=100, nj_lo=3, nj_hi=10, b=16, tau=10.0, tol=1e-6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pipeline", "pipeline", "build", "apply", "apply", "apply", "solve", "arnoldi", "direct",
                       "batched"])
    if kind == "batched":
        return dict(kind=kind, prec=rng.choice(["f64", "f64_tc"]), count=rng.randint(4, 24),
                    shapes=rng.randrange(1 << 20), d_lo=512, d_hi=16384, k_lo=5, k_hi=60, nj_lo=3, nj_hi=10,
                    b=rng.choice([4, 8, 16]), tau=10.0, tol=1e-6)
    d = _log_int(rng, 250, 65536)
    if rng.random() < 0.3:
        d = max(256, d // 256 * 256)
    # few classes on small images, up to 200 on the largest; plain FP64 and the eigensolver-bound calls stay at sizes
    # below the largest listed cases
    k = _log_int(rng, 4, max(8, min(200, d // 40)))
    nj_lo = rng.randint(3, 8)
    nj_hi = nj_lo + rng.choice([0, 0, 1, 2])
    case = dict(kind=kind, d=d, k=k, nj_lo=nj_lo, nj_hi=nj_hi, tau=10.0)
    if kind == "apply":
        case["prec"] = rng.choice(["f64", "f64_tc", "bf16", "bf16", "f32"])
        case["op"] = rng.choice(["SW", "SB", "M"] + (["N"] if case["prec"] in ("f64", "f64_tc") else []))
        case["b"] = rng.choice([1, 2, 3, 4, 7, 8, 13, 16, 20, 29, 32])
        return case
    if kind in ("build", "solve", "arnoldi", "direct"):
        case["k"] = min(k, 120)
    case["prec"] = rng.choice(["f64", "f64_tc"]) if case["d"] * case["k"] < (1 << 21) else "f64_tc"
    case["b"] = rng.choice([2, 4, 8, 16]) if case["k"] > 8 else rng.choice([1, 2])
    if kind in ("pipeline", "solve", "arnoldi"):
        case["tol"] = 1e-6
    if kind != "build":
        case["t"] = case["k"] - 1
    if kind == "pipeline":
        case["test"] = rng.randint(2, 6)
    if kind in ("pipeline", "build"):
        case["x"] = rng.choice(["f64", "f64", "f32"])
    return case


# ------------------------------------------------------------------------------------------------ inputs

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _counts(case, shape_seed):
    r = random.Random(shape_seed)
    return [r.randint(case["nj_lo"], case["nj_hi"]) for _ in range(case["k"])]


def _samples(d, counts, gen, test=0, dtype=torch.float64):
    """(X (n, d), labels (n,), held-out (k test, d)) of class clusters; labels shuffled."""
    dev = _device()
    k = len(counts)
    means = torch.randn(k, d, dtype=torch.float64, device=dev, generator=gen)
    lab = torch.repeat_interleave(torch.arange(k, device=dev), torch.tensor(counts, device=dev))
    lab = lab[torch.randperm(lab.numel(), device=dev, generator=gen)]

    def of(which):
        x = torch.randn(which.numel(), d, dtype=torch.float64, device=dev, generator=gen)
        return x.mul_(0.3).add_(means[which]).clamp_(0.0, 1.0)

    X = of(lab).to(dtype).contiguous()
    held = of(torch.repeat_interleave(torch.arange(k, device=dev), test)) if test else None
    return X, lab.to(torch.int32), held


def _generator(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed))
    return g


def _config(case):
    return eda.config(prec=PREC[case["prec"]], block_b=case["b"], tau=case["tau"], m_form=1)


def _batch_shapes(case):
    r = random.Random(case["shapes"])
    out = []
    for _ in range(case["count"]):
        d = _log_int(r, case["d_lo"], case["d_hi"])
        k = min(r.randint(case["k_lo"], case["k_hi"]), max(3, d // 20))
        out.append((d, [r.randint(case["nj_lo"], case["nj_hi"]) for _ in range(k)]))
    return out


def _inputs(case, seed):
    """What the user has before any call of the library (no handle)."""
    gen = _generator(seed)
    if case["kind"] == "batched":
        probs = []
        for d, counts in _batch_shapes(case):
            X, lab, _ = _samples(d, counts, gen)
            probs.append(dict(X=X, labels=lab, k=len(counts), t=len(counts) - 1, tol=case["tol"]))
        return dict(case=case, probs=probs)
    dtype = torch.float32 if case.get("x") == "f32" else torch.float64
    X, lab, held = _samples(case["d"], _counts(case, case["d"] * 1000 + case["k"]), gen, case.get("test", 0), dtype)
    s = dict(case=case, X=X, labels=lab, held=held)
    if case["kind"] == "apply":
        low = case["prec"] in ("f32", "bf16")
        s["block"] = torch.randn(case["b"], case["d"], dtype=torch.float32 if low else torch.float64, device=X.device,
                                 generator=gen)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["cfg"] = _config(case)
    if case["kind"] not in ("pipeline", "build", "batched"):
        s["h"] = eda.build(s["X"], s["labels"], case["k"], s["cfg"])
    if case["kind"] == "apply":
        h = s["h"]
        s["alpha"] = {"SW": -0.5 * h.c2, "SB": h.c2}.get(case["op"], 0.0)
    return s


# ------------------------------------------------------------------------------------------------ one pass

def _converged(code):
    if code != 0:
        raise RuntimeError(f"the solve ended with status {code}")


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "pipeline":
        with eda.build(state["X"], state["labels"], case["k"], state["cfg"]) as h:
            V, lam, _, _, code = h.solve(case["t"], case["tol"])
            _converged(code)
            return {"V": V, "lam": lam, "P": h.project(V, state["held"])}
    if kind == "build":
        with eda.build(state["X"], state["labels"], case["k"], state["cfg"]) as h:
            out = h.factors()
            out.pop("has_labels")
            return out
    if kind == "apply":
        return state["h"].apply_exp(OPS[case["op"]], state["block"], alpha=state["alpha"])
    if kind == "solve":
        V, lam, Y, _, code = state["h"].solve(case["t"], case["tol"], want_y=True)
        _converged(code)
        return {"V": V, "lam": lam, "Y": Y}
    if kind == "arnoldi":
        V, lam, _, code = state["h"].solve_arnoldi(case["t"], case["tol"])
        _converged(code)
        return {"V": V, "lam": lam}
    if kind == "direct":
        V, lam, _, _ = state["h"].solve_direct(case["t"])
        return {"V": V, "lam": lam}
    res, code = eda.solve_batched(state["probs"], state["cfg"])
    _converged(code)
    return [(r["V"], r["lam"]) for r in res]


# ------------------------------------------------------------------------------------------------ the work of a pass

def _work_of(kind, prec, d, n, k, b, t, m, xbytes, op="M"):
    """Bytes read and written once and floating-point operations of the definition (FP64 ones, also where they are done
    as several products of another type)."""
    nk = n + k
    gram = d * (n * (n + 1.0) + k * (k + 1.0))
    small = 10.0 * (float(n) ** 3 + float(k) ** 3)          # the Grams' eigenpairs or the squaring
    m_apply = 4.0 * d * nk * b + 2.0 * b * (3.0 * n * n + 2.0 * n * k + k * k)
    if kind == "apply":
        es = {"f64": 8, "f64_tc": 8, "f32": 4, "bf16": 2}[prec]
        xs = 8 if prec in ("f64", "f64_tc") else 4
        w = {"SW": n, "SB": k}.get(op, nk)
        flops = (4.0 * d * w * b + 2.0 * w * w * b) if op in ("SW", "SB") else m_apply
        return dict(bytes=float(es * d * w + 8 * w * w + 2 * xs * d * b), flops=flops)
    blocks = math.ceil(t / b) + 2 if t else 0
    krylov = blocks * m_apply + 4.0 * d * b * b * blocks * (blocks + 1.0)
    finish = 4.0 * d * n * t + 2.0 * float(n) * n * t + 6.0 * d * t * t
    if kind == "build":
        return dict(bytes=float(xbytes * d * n + 8 * d * nk + 16 * (n * n + k * k) + 8 * nk + 4 * nk),
                    flops=gram + small + 3.0 * d * n)
    if kind in ("solve", "arnoldi"):
        return dict(bytes=float(8 * d * nk + 8 * (n * n + k * k) + 8 * d * t * (2 if kind == "solve" else 1)),
                    flops=krylov + finish)
    if kind == "direct":
        return dict(bytes=float(8 * d * nk + 8 * (n * n + k * k) + 8 * d * t),
                    flops=(4.0 / 3.0 + 6.0) * float(n) ** 3 + 2.0 * d * nk * t + 4.0 * d * t * t)
    return dict(bytes=float(xbytes * d * n + 8 * d * (t + m)) + 8.0 * t * (m + 1),
                flops=gram + small + krylov + finish + 2.0 * d * t * m)


def work(case):
    if case["kind"] == "batched":
        parts = [_work_of("pipeline", case["prec"], d, sum(c), len(c), case["b"], len(c) - 1, 0, 8)
                 for d, c in _batch_shapes(case)]
        return dict(bytes=sum(p["bytes"] for p in parts), flops=sum(p["flops"] for p in parts))
    n = sum(_counts(case, case["d"] * 1000 + case["k"]))
    return _work_of(case["kind"], case["prec"], case["d"], n, case["k"], case["b"], case.get("t", 0),
                    case.get("test", 0) * case["k"], 4 if case.get("x") == "f32" else 8, case.get("op", "M"))


# ------------------------------------------------------------------------------------------------ 64-bit values

def _factors(X, lab, k):
    """H_W, H_B as (columns, d) tensors, the class counts and the class-major order, from the definitions."""
    X = X.double()
    lab = lab.long()
    counts = torch.bincount(lab, minlength=k)
    mu_j = torch.zeros(k, X.shape[1], dtype=torch.float64, device=X.device).index_add_(0, lab, X)
    mu_j /= counts.double()[:, None]
    perm = torch.argsort(lab, stable=True)
    HW = X[perm] - mu_j[lab[perm]]
    HB = counts.double().sqrt()[:, None] * (mu_j - X.mean(0))
    return HW, HB, counts, perm


def _k_of(G, alpha):
    """alpha phi(alpha G), phi(z) = (e^z - 1) / z."""
    w, Q = torch.linalg.eigh(G)
    z = alpha * w.clamp(min=0.0)
    phi = torch.where(z.abs() > 1e-300, torch.expm1(z) / torch.where(z == 0, torch.ones_like(z), z),
                      torch.ones_like(z))
    return (Q * (alpha * phi)) @ Q.T, w


def _eigenvalues(HW, HB, c2, t):
    """The t largest eigenvalues of exp(-c2 S_W / 2) exp(c2 S_B) exp(-c2 S_W / 2) = I + Z C Z^T, Z = [H_W H_B]."""
    n, k = HW.shape[0], HB.shape[0]
    Z = torch.cat([HW, HB])
    G = Z @ Z.T
    A1 = torch.zeros_like(G)
    A2 = torch.zeros_like(G)
    A1[:n, :n] = _k_of(G[:n, :n], -0.5 * c2)[0]
    A2[n:, n:] = _k_of(G[n:, n:], c2)[0]

    def times(a, b):
        return a + b + a @ G @ b

    C = times(times(A1, A2), A1)
    w, Q = torch.linalg.eigh(G)
    R = Q * w.clamp(min=0.0).sqrt()
    return 1.0 + torch.linalg.eigvalsh(R.T @ (0.5 * (C + C.T)) @ R).flip(0)[:t]


def _scale(HW, HB, tau):
    return tau / max(torch.linalg.eigvalsh(H @ H.T)[-1].item() for H in (HW, HB))


def exact(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "batched":
        out = []
        for p in s["probs"]:
            HW, HB, _, _ = _factors(p["X"], p["labels"], p["k"])
            out.append((None, _eigenvalues(HW, HB, _scale(HW, HB, case["tau"]), p["t"])))
        return out
    HW, HB, counts, perm = _factors(s["X"], s["labels"], case["k"])
    c2 = _scale(HW, HB, case["tau"])
    if case["kind"] == "build":
        KW, ew = _k_of(HW @ HW.T, -0.5 * c2)
        KB, eb = _k_of(HB @ HB.T, c2)
        return dict(HW=HW, HB=HB, counts=counts.to(torch.int32), perm=perm.to(torch.int32), GW=HW @ HW.T, GB=HB @ HB.T,
                    KW=KW, KB=KB, evals_w=ew, evals_b=eb)
    if case["kind"] == "apply":
        X = s["block"].double()

        def exp_apply(H, alpha, Y):
            return Y + ((Y @ H.T) @ _k_of(H @ H.T, alpha)[0]) @ H

        if case["op"] == "SW":
            return exp_apply(HW, -0.5 * c2, X)
        if case["op"] == "SB":
            return exp_apply(HB, c2, X)
        if case["op"] == "N":
            return exp_apply(HW, -c2, exp_apply(HB, c2, X))
        return exp_apply(HW, -0.5 * c2, exp_apply(HB, c2, exp_apply(HW, -0.5 * c2, X)))
    # the eigenvectors' signs are free, so V, Y and P have no value of their own
    out = {"V": None, "lam": _eigenvalues(HW, HB, c2, case["t"])}
    if case["kind"] == "pipeline":
        out["P"] = None
    if case["kind"] == "solve":
        out["Y"] = None
    return out
