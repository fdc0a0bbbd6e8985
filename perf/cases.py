"""What the speed of this repository is measured on.

A case is one pass of the work that users of the library have it do, through
its public entry points (`paper_2101_06599_gb300.de`):

  run      a whole optimisation job on one population: the initial population
           is given from page-locked host memory, evaluated, advanced by
           `gens` generations, and the best row, the population and its
           fitness come back to the host;
  large    a running optimisation of the largest populations, which no cache
           holds: `gens` further generations, then the state to the host;
  rotated  a job as `run` on a shifted-rotated objective, the product in FP32
           or on the tensor cores;
  batch    `gens` further generations of many independent instances of uneven
           sizes, then every population to the host;
  lent     one generation on device buffers that the caller owns.

Sizes are those of workloads.py (its five workloads, at fewer generations),
of the published runs (Table II) and of the tests.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2101_06599_gb300 import de as DE
from paper_2101_06599_gb300 import workloads as W

BOXES = {k: (float(v[0]), float(v[1])) for k, v in W.BOXES.items()}


def listed():
    return [
        # the smallest population (100 x 30), one generation at a time inside a program that owns the buffers
        dict(name="lent_sphere_100x30", kind="lent", N=100, D=30, obj="sphere", F=0.5, CR=0.9),
        # the same call on rows longer than L2 holds, an odd D (a test's), a pitch that is not D
        dict(name="lent_rosenbrock_8192x4097", kind="lent", N=8192, D=4097, obj="rosenbrock", F=0.5, CR=0.9),
        # the plain job: sphere, 100 x 30, 200 generations
        dict(name="run_sphere_100x30_nec", kind="run", N=100, D=30, obj="sphere", xo="nec", F=0.5, CR=0.9, gens=200),
        # a published run (Griewank, D = 500, Np = 300, F = 0.25, Cr = 0.45), binomial crossover
        dict(name="run_griewank_300x500_bin", kind="run", N=300, D=500, obj="griewank", xo="bin", F=0.25, CR=0.45,
             gens=200),
        # the large-scale job that still sits in L2, new exponential crossover at a high rate
        dict(name="run_rastrigin_1024x1000_nec", kind="run", N=1024, D=1000, obj="rastrigin", xo="nec", F=0.5, CR=0.9,
             gens=200),
        # the same job with the classic exponential crossover at the middle rate
        dict(name="run_rastrigin_1024x1000_exp", kind="run", N=1024, D=1000, obj="rastrigin", xo="exp", F=0.5, CR=0.5,
             gens=100),
        # the largest populations, the objective and crossover that the library is quoted on
        dict(name="large_rosenbrock_16384x10000_nec", kind="large", N=16384, D=10000, obj="rosenbrock", xo="nec",
             F=0.5, CR=0.9, gens=100),
        # the same size at its costliest: Ackley, binomial
        dict(name="large_ackley_16384x10000_bin", kind="large", N=16384, D=10000, obj="ackley", xo="bin", F=0.5,
             CR=0.9, gens=16),
        # independent instances, D log-uniform in [10, 2000], four objectives
        dict(name="batch_128", kind="batch", n=128, xo="nec", F=0.5, CR=0.9, gens=100),
        # shifted-rotated objectives at their workload's size, once in each precision of the product
        dict(name="rotated_rastrigin_4096x1024_fp16", kind="rotated", N=4096, D=1024, obj="sr_rastrigin", xo="nec",
             F=0.5, CR=0.9, prec="fp16", gens=50),
        dict(name="rotated_elliptic_4096x1024_bf16", kind="rotated", N=4096, D=1024, obj="sr_elliptic", xo="nec",
             F=0.5, CR=0.9, prec="bf16", gens=50),
        dict(name="rotated_rastrigin_4096x1024_fp32", kind="rotated", N=4096, D=1024, obj="sr_rastrigin", xo="nec",
             F=0.5, CR=0.9, prec="fp32", gens=20),
    ]


# Runs are short enough for the 64-bit results to stay on the same course: a
# selection between two nearly equal values that FP32 takes the other way
# changes a row, and later the rows that use it as a donor.
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "lent", "large", "batch", "rotated", "rotated"])
    F, CR = round(rng.uniform(0.25, 0.8), 3), round(rng.uniform(0.1, 0.95), 3)
    if kind == "run":
        N = _log_int(rng, 20, 2000)
        D = _log_int(rng, 8, min(2000, 2_000_000 // N))
        return dict(kind=kind, N=N, D=D, F=F, CR=CR, xo=rng.choice(["nec", "exp", "bin"]), gens=rng.randint(20, 80),
                    obj=rng.choice(["sphere", "rastrigin", "ackley", "rosenbrock", "griewank"]))
    if kind == "lent":
        N = _log_int(rng, 50, 10000)
        return dict(kind=kind, N=N, D=_log_int(rng, 10, min(10000, 40_000_000 // N)), F=F, CR=CR,
                    obj=rng.choice(["sphere", "rastrigin", "ackley", "rosenbrock", "elliptic"]))
    if kind == "large":
        return dict(kind=kind, N=_log_int(rng, 2000, 16384), D=_log_int(rng, 2048, 10000), F=F, CR=CR,
                    xo=rng.choice(["nec", "exp", "bin"]), obj=rng.choice(["rosenbrock", "ackley", "rastrigin"]),
                    gens=rng.randint(8, 20))
    if kind == "batch":
        return dict(kind=kind, n=_log_int(rng, 16, 128), xo="nec", F=F, CR=CR, gens=rng.randint(10, 60))
    prec = rng.choice(["fp32", "bf16", "fp16"])
    return dict(kind=kind, N=_log_int(rng, 500, 4096), D=rng.randint(64, 1024) if prec == "fp32" else
                256 * rng.randint(1, 4), F=F, CR=CR, xo="nec", obj=rng.choice(["sr_rastrigin", "sr_elliptic"]),
                prec=prec, gens=rng.randint(10, 50))


def _uniform(N, D, box, seed):
    """A seeded uniform N x D population in the box, made on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    x = torch.rand((N, D), generator=g, device="cuda", dtype=torch.float32)
    return (box[0] + (box[1] - box[0]) * x).clamp_(box[0], box[1])


def _host(*shape):
    return torch.empty(shape, dtype=torch.float32, pin_memory=True)


def _rotation_params(case, seed):
    return dict(shift=W.shift_vector(case["D"], seed=seed), rotation=W.rotation(case["D"], seed=seed + 1),
                prec=case["prec"])


def _batch_specs(case):
    return [dict(N=s.N, D=s.D, obj=s.objective, bounds=BOXES[s.objective], xo=case["xo"], CR=case["CR"], F=case["F"])
            for s in W.batched_specs(case["n"])]


def prepare(case, seed):
    kind, s = case["kind"], dict(case=dict(case), seed=int(seed))
    if kind == "lent":
        N, D = case["N"], case["D"]
        pitch = 4 * ((D + 3) // 4)
        x = torch.zeros((N, pitch), device="cuda")
        x[:, :D] = _uniform(N, D, BOXES[case["obj"]], seed)
        s.update(pitch=pitch, x=x, f=_objective(case["obj"], x[:, :D]).float(), x_out=torch.zeros_like(x),
                 f_out=torch.empty(N, device="cuda"), gen=0)
        return s
    if kind == "batch":
        specs = _batch_specs(case)
        s["opt"] = DE.Batch(specs, seed=seed)
        s["x"], s["f"] = _host(sum(p["N"] * p["D"] for p in specs)), _host(sum(p["N"] for p in specs))
        s["views"], a, b = [], 0, 0
        for p in specs:
            s["views"].append((s["x"][a:a + p["N"] * p["D"]], s["f"][b:b + p["N"]]))
            a, b = a + p["N"] * p["D"], b + p["N"]
    else:
        N, D = case["N"], case["D"]
        params = _rotation_params(case, seed) if kind == "rotated" else None
        s["opt"] = DE.Optimizer(N, D, F=case["F"], CR=case["CR"], xo=case["xo"], obj=case["obj"],
                                bounds=BOXES[case["obj"]], seed=seed, params=params)
        s["x"], s["f"], s["best"] = _host(N, D), _host(N), _host(D)
        if kind != "large":
            s["x0"] = _host(N, D)
            s["x0"].copy_(_uniform(N, D, BOXES[case["obj"]], seed))
            s["start"] = s["x0"].numpy()
    s["opt"].prepare_run(case["gens"])   # a program that repeats a run keeps its plan
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "lent":
        DE.de_nec_step_noalloc(s["x"].data_ptr(), s["f"].data_ptr(), s["x_out"].data_ptr(), s["f_out"].data_ptr(),
                               case["N"], case["D"], s["pitch"], case["F"], case["CR"], case["obj"],
                               BOXES[case["obj"]], s["seed"], s["gen"], torch.cuda.current_stream().cuda_stream)
        s["gen"] += 1
        return {"x": s["x_out"][:, :case["D"]], "f": s["f_out"]}
    opt = s["opt"]
    if kind in ("run", "rotated"):
        opt.set_population(s["start"])
    opt.run(case["gens"])
    if kind == "batch":
        for k, (x, f) in enumerate(s["views"]):
            DE.de_batch_get_population(opt.ctx, k, x, f)
        return {"x": s["x"], "f": s["f"]}
    f, _, _ = DE.de_best(opt.ctx, s["best"])
    DE.de_get_population(opt.ctx, s["x"], s["f"])
    return {"x": s["x"], "f": s["f"], "best_x": s["best"], "best_f": np.float32(f)}


_FLOPS = {"sphere": 2, "rastrigin": 18, "ackley": 18, "rosenbrock": 7, "griewank": 30, "elliptic": 4,
          "sr_rastrigin": 20, "sr_elliptic": 4}   # of one gene's term
_L2 = 126e6


def _per_generation(N, D, obj, xo, CR):
    """Bytes and operations of one generation out of memory: the parents, three
    donors of every gene that crosses, and the rows of the trials that win (a
    quarter of them, about what the early generations show)."""
    share = CR if xo == "bin" else min(1.0, (1.0 - CR ** D) / ((1.0 - CR) * D))
    return 4.0 * N * D * (1 + 3 * share + 0.25), N * D * (_FLOPS[obj] + 3 * share)


def work(case):
    kind = case["kind"]
    if kind == "lent":
        return {"bytes": 8.0 * case["N"] * (case["D"] + 1),
                "flops": _per_generation(case["N"], case["D"], case["obj"], "nec", case["CR"])[1]}
    specs = _batch_specs(case) if kind == "batch" else [case]
    total = {"bytes": 0.0, "flops": 0.0}
    held = sum(4.0 * p["N"] * p["D"] for p in specs)
    for p in specs:
        b, f = _per_generation(p["N"], p["D"], p["obj"], p["xo"], p["CR"])
        if kind == "rotated":
            f += 2.0 * p["N"] * p["D"] * p["D"]
        total["flops"] += f * case["gens"]
        # what L2 holds has to be read and written once in all
        total["bytes"] += b * case["gens"] if held > _L2 / 2 else 8.0 * p["N"] * (p["D"] + 1)
    return total


# ---- the same results in plain torch -------------------------------------------
# Draws and trial genes are defined bit by bit (Philox4x32-10; x1 + F (x2 - x3)
# with each operation rounded to FP32); fitness and selection are in 64 bits.
_M32 = 0xFFFFFFFF


def _philox(seed, stream, inst, gen, row, block):
    """Philox4x32-10 (Salmon et al. 2011) words at counter (block, row, gen,
    stream << 24 | inst), as four int64 tensors."""
    c0, c1, c2, c3 = torch.broadcast_tensors(torch.as_tensor(block, device="cuda"), torch.as_tensor(row, device="cuda"),
                                             torch.as_tensor(gen, device="cuda"),
                                             torch.as_tensor(inst, device="cuda") + (stream << 24))
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((b >> 32) & _M32) ^ c1 ^ k0, b & _M32, ((a >> 32) & _M32) ^ c3 ^ k1, a & _M32
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _donors(seed, inst, gen, row, N, D):
    """r1, r2, r3 distinct and not the row, and j_rand: each a multiply-shift of
    its word, stepped over the rows already taken in ascending order."""
    w = _philox(seed, 1, inst, gen, row, 0)
    taken, out = [row.clone()], []
    for k in range(3):
        v = (w[k] * (N - 1 - k)) >> 32
        for e in torch.stack(taken).sort(0).values:
            v = v + (v >= e)
        taken.append(v)
        out.append(v)
    return out + [(w[3] * D) >> 32]


def _lengths(seed, inst, gen, row, D, xo, CR):
    """Segment lengths: smallest n with Cr^n <= U (nec), or Alg. 8's walk (exp)."""
    if xo == "nec":
        w = _philox(seed, 2, inst, gen, row, 0)[0]
        top = int(D.max()) if torch.is_tensor(D) else D
        T = np.ceil(np.multiply.accumulate(np.full(max(1, top), CR)) * 4294967296.0)
        T = torch.from_numpy(np.ascontiguousarray(T[T > 1][::-1].astype(np.int64))).cuda()   # ascending
        L = 1 + T.numel() - torch.searchsorted(T, w, right=True)
        L = torch.where(w == 0, torch.full_like(L, top), L)
        return torch.minimum(L, torch.as_tensor(D, device="cuda"))
    t, k = math.ceil(CR * 4294967296.0), 0
    L, on = torch.ones_like(row), torch.ones_like(row, dtype=torch.bool)
    while 4 * k < D and bool(on.any()):
        for w in _philox(seed, 4, inst, gen, row, k):
            on = on & (w < t) & (L < D)
            L = L + on
        k += 1
    return L


def _objective(obj, x, params=None):
    """FP64 value of each row of x."""
    x = x.double()
    D = x.shape[1]
    if params is not None:
        x = (x - params[0]) @ params[1].T
        obj = obj[3:]
    if obj == "sphere":
        return (x * x).sum(1)
    if obj == "rastrigin":
        return (x * x - 10 * torch.cos(2 * math.pi * x)).sum(1) + 10 * D
    if obj == "ackley":
        return (-20 * torch.exp(-0.2 * (x * x).mean(1).sqrt()) - torch.exp(torch.cos(2 * math.pi * x).mean(1))
                + 20 + math.e)
    if obj == "rosenbrock":
        a, b = x[:, :-1], x[:, 1:]
        return (100 * (a * a - b) ** 2 + (1 - a) ** 2).sum(1)
    j = torch.arange(D, device=x.device, dtype=torch.float64)
    if obj == "griewank":
        return (x * x).sum(1) / 4000 - torch.cos(x / (j + 1).sqrt()).prod(1) + 1
    return (torch.pow(10.0, 6 * j / max(1, D - 1)) * x * x).sum(1)


def _generation(x, f, spec, seed, gen, inst=0, params=None, drawn=None):
    """One generation of an FP32 population x with FP64 fitness f."""
    N, D = x.shape
    lo, hi = (torch.tensor(v, dtype=torch.float32, device="cuda") for v in BOXES[spec["obj"]])
    F = torch.tensor(spec["F"], dtype=torch.float32, device="cuda")
    j = torch.arange(D, device="cuda", dtype=torch.int32)
    new_x, new_f = x.clone(), f.clone()
    step = max(1, 8_000_000 // D)
    for a in range(0, N, step):
        row = torch.arange(a, min(N, a + step), device="cuda")
        at = slice(a, a + len(row))
        r1, r2, r3, jr = _donors(seed, inst, gen, row, N, D) if drawn is None else [v[at] for v in drawn[:4]]
        if spec["xo"] == "bin":
            q = torch.arange((D + 3) // 4, device="cuda")
            w = torch.stack(_philox(seed, 3, inst, gen, row[:, None], q[None, :]), -1).reshape(len(row), -1)[:, :D]
            mask = (w < math.ceil(spec["CR"] * 4294967296.0)) | (j == jr[:, None])
        else:
            L = _lengths(seed, inst, gen, row, D, spec["xo"], spec["CR"]) if drawn is None else drawn[4][at]
            mask = (j - jr[:, None].int()) % D < L[:, None].int()
        v = torch.clamp(x[r1] + F * (x[r2] - x[r3]), lo, hi)
        v = torch.where(mask, v, x[at])
        fv = _objective(spec["obj"], v, params)
        win = fv < f[at]
        new_x[at] = torch.where(win[:, None], v, x[at])
        new_f[at] = torch.where(win, fv, f[at])
    return new_x, new_f


def _initial(N, D, box, seed, inst=0):
    """The uniform population that a context starts from."""
    lo, hi = (torch.tensor(v, dtype=torch.float32, device="cuda") for v in box)
    q, out = torch.arange((D + 3) // 4, device="cuda"), torch.empty((N, D), device="cuda")
    step = max(1, 8_000_000 // D)
    for a in range(0, N, step):
        row = torch.arange(a, min(N, a + step), device="cuda")
        w = torch.stack(_philox(seed, 0, inst, 0, row[:, None], q[None, :]), -1).reshape(len(row), -1)[:, :D]
        out[a:a + len(row)] = torch.clamp(lo + (hi - lo) * ((w >> 8).float() * 2.0 ** -24), lo, hi)
    return out


def _values(obj, x, params=None):
    step = max(1, 8_000_000 // x.shape[1])
    return torch.cat([_objective(obj, x[a:a + step], params) for a in range(0, x.shape[0], step)])


def exact(case, seed):
    kind, seed = case["kind"], int(seed)
    if kind == "batch":
        specs, xs, fs = _batch_specs(case), [], []
        for k, p in enumerate(specs):
            xs.append(_initial(p["N"], p["D"], p["bounds"], seed, inst=k))
            fs.append(_values(p["obj"], xs[k]))
        size = torch.tensor([p["N"] for p in specs], device="cuda")
        inst = torch.repeat_interleave(torch.arange(len(specs), device="cuda"), size)
        row = torch.cat([torch.arange(p["N"], device="cuda") for p in specs])
        N = torch.repeat_interleave(size, size)
        D = torch.repeat_interleave(torch.tensor([p["D"] for p in specs], device="cuda"), size)
        at = [0] + size.cumsum(0).tolist()
        for g in range(case["gens"]):
            drawn = _donors(seed, inst, g, row, N, D) + [_lengths(seed, inst, g, row, D, case["xo"], case["CR"])]
            for k, p in enumerate(specs):
                xs[k], fs[k] = _generation(xs[k], fs[k], p, seed, g, k, None, [v[at[k]:at[k + 1]] for v in drawn])
        return {"x": torch.cat([x.reshape(-1).double() for x in xs]), "f": torch.cat(fs)}
    N, D, params = case["N"], case["D"], None
    if kind == "lent":
        x = _uniform(N, D, BOXES[case["obj"]], seed)
        f = _values(case["obj"], x).float()
        x, f = _generation(x, f.double(), dict(case, xo="nec"), seed, 0)
        return {"x": x.double(), "f": f}
    if kind == "rotated":
        p = _rotation_params(case, seed)
        params = [torch.from_numpy(p[k]).cuda().double() for k in ("shift", "rotation")]
    x = _initial(N, D, BOXES[case["obj"]], seed) if kind == "large" else _uniform(N, D, BOXES[case["obj"]], seed)
    f = _values(case["obj"], x, params)
    for g in range(case["gens"]):
        x, f = _generation(x, f, case, seed, g, params=params)
    k = int(f.argmin())
    return {"x": x if kind == "large" else x.double(), "f": f, "best_x": x[k].double(), "best_f": f[k]}
