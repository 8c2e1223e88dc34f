"""The workloads this library is timed on.

Each case is one pass through the public entry points as a program that uses
the library makes it: a time step (fmm_build + fmm_evaluate), a solver's
matrix-vector product on a fixed tree (new charges + evaluate), the weighted
energy with its gradients, a batch of independent systems, and the
allocation-free Morton sort. Sizes, orders and options are those of the
library's own configurations, tests and benchmark, and the ranges between them.

A case is a dict of plain values:
  kind       "step", "matvec", "energy", "batch" or "sort"
  n          particles (of the whole batch for "batch")
  dist       "uniform": uniform cube, charges U[-1, 1]; "plummer": Plummer
             sphere truncated at r = 20, charges U[0, 1] / n; "both" ("batch"
             only): every other system a Plummer sphere, charges U[-1, 1]
  p, theta, ncrit, precision   of the handle
  dtype      "f32" or "f64" particles
  host       particles and results in host arrays ("step" only)
  systems    number of systems ("batch" only), sizes log-uniform
"""
import ctypes
import math

import numpy as np
import torch

from paper_1106_2176_gb300 import FMM
from paper_1106_2176_gb300.autograd import fmm_energy
from paper_1106_2176_gb300.batch import FMMBatch
from paper_1106_2176_gb300.fmm import FMM_F32, FMM_F64, lib

DTYPES = {"f32": torch.float32, "f64": torch.float64}
EXACT_MAX_PAIRS = 9e10  # direct sums beyond this many pairs take too long to repeat


def _case(name, kind, n, dist="uniform", p=8, theta=0.5, ncrit=64, precision="mixed", dtype="f32", host=False,
          systems=1):
    c = dict(kind=kind, n=n, dist=dist, p=p, theta=theta, ncrit=ncrit, precision=precision, dtype=dtype, host=host,
             systems=systems)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # A small system stepped in time: the smallest size of the batching
        # workload, where launches and host synchronisations set the pace.
        _case("step_1k", "step", 1000, p=6),
        # The basic configuration (N = 16,384, p = 6, theta = 0.5) in mixed
        # precision on double-precision particles, as a double-precision
        # simulation code hands them over.
        _case("step_16k_f64in", "step", 16384, p=6, dtype="f64"),
        # The same method at a higher order and a stricter acceptance test (the
        # precision study's p = 10, theta = 0.4), at a ragged size.
        _case("step_100k_p10", "step", 100003, p=10, theta=0.4),
        # A clustered system stepped in time: deep adaptive tree, pairs across
        # levels.
        _case("step_1m_plummer", "step", 1000000, dist="plummer"),
        # The headline workload: N = 10^7 uniform, FP32, p = 8, the tuned leaf size.
        _case("step_10m", "step", 10000000, ncrit=128),
        # Particles and results in host memory, as a caller without a GPU array
        # of its own has them.
        _case("step_300k_host", "step", 300007, host=True),
        # Every stage in FP64: the reference path of an accuracy study.
        _case("step_50k_fp64", "step", 50000, precision="fp64", dtype="f64"),
        # High order past the tensor-core engine (rotation-based translations),
        # mixed precision.
        _case("step_60k_p16", "step", 60001, p=16),
        # A solver's matrix-vector product: new charges on a fixed tree.
        _case("matvec_1m_p10", "matvec", 1000000, p=10),
        # Energy and its gradients (training, variational problems): forward
        # and backward through autograd on the clustered distribution.
        _case("energy_1m_plummer", "energy", 1000000, dist="plummer"),
        # Many independent systems of uneven size evaluated together (sizes
        # log-uniform in [10^3, 2 10^4], half of them clustered).
        _case("batch_32", "batch", 32 * 6342, dist="both", p=6, ncrit=128, systems=32),
        # Keys and sorting permutation for a caller that cannot allocate.
        _case("sort_1m", "sort", 1000003),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step_f64in", "host", "fp64", "highp", "matvec", "energy", "batch", "sort"])
    dist = rng.choice(["uniform", "plummer"])
    ncrit = rng.choice([32, 64, 100, 128])
    theta = rng.choice([0.4, 0.5, 0.6])
    p = rng.randint(4, 10)
    if kind in ("step", "step_f64in"):
        return _case(None, "step", _log_int(rng, 1000, 1500000), dist, p, theta, ncrit,
                     dtype="f32" if kind == "step" else "f64")
    if kind == "host":
        return _case(None, "step", _log_int(rng, 10000, 1000000), dist, p, theta, ncrit, host=True)
    if kind == "fp64":
        return _case(None, "step", _log_int(rng, 1000, 50000), dist, rng.randint(4, 8), 0.5, 64, "fp64", "f64")
    if kind == "highp":
        return _case(None, "step", _log_int(rng, 1000, 60000), dist, rng.randint(12, 16), 0.5, 64)
    if kind == "matvec":
        return _case(None, "matvec", _log_int(rng, 1000, 1000000), dist, p, theta, ncrit)
    if kind == "energy":
        return _case(None, "energy", _log_int(rng, 1000, 1000000), dist, p, theta, ncrit)
    if kind == "batch":
        s = rng.randint(8, 32)
        return _case(None, "batch", s * 6342, "both", p, 0.5, ncrit, systems=s)
    return _case(None, "sort", _log_int(rng, 1000, 1048576), dist, dtype=rng.choice(["f32", "f64"]))


# -- inputs -------------------------------------------------------------------

def _particles(case, n, dist, g):
    """Positions, charges and weights on the GPU in the case's type."""
    kw = dict(generator=g, device="cuda", dtype=torch.float64)
    if dist == "uniform":
        x = torch.rand(n, 3, **kw) * 2 - 1
        q = torch.rand(n, **kw) * 2 - 1
    else:
        # radii by inversion of the Plummer mass profile cut off at r = 20
        u = (torch.rand(n, **kw) * (20.0 ** 3 / (1 + 20.0 ** 2) ** 1.5)).clamp_min(1e-12)
        r = 1 / torch.sqrt(u ** (-2.0 / 3.0) - 1)
        ct = torch.rand(n, **kw) * 2 - 1
        st = torch.sqrt(1 - ct * ct)
        ph = torch.rand(n, **kw) * (2 * math.pi)
        x = torch.stack([r * st * torch.cos(ph), r * st * torch.sin(ph), r * ct], 1)
        q = torch.rand(n, **kw) / n if case["kind"] != "batch" else torch.rand(n, **kw) * 2 - 1
    w = torch.randn(n, **kw) if case["kind"] == "energy" else None
    dt = DTYPES[case["dtype"]]
    return x.to(dt).contiguous(), q.to(dt), None if w is None else w.to(dt)


def _sizes(case, seed):
    """System sizes of a batch: log-uniform in [10^3, 2 10^4], the first ones of every seed the same."""
    s = case["systems"]
    t = (np.arange(s) + 0.5) / s
    order = np.random.default_rng(7).permutation(s)
    return [int(1000 * 20 ** v) + (i * 13) % 7 for i, v in enumerate(t[order])]


def _inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + 17)
    if case["kind"] == "batch":
        return [_particles(case, n, "plummer" if i % 2 else "uniform", g)[:2] for i, n in enumerate(_sizes(case, seed))]
    return _particles(case, case["n"], case["dist"], g)


def _handle(case):
    return FMM(case["n"], p=case["p"], theta=case["theta"], ncrit=case["ncrit"], precision=case["precision"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return dict(case=case, batch=FMMBatch(_inputs(case, seed), p=case["p"], theta=case["theta"], ncrit=case["ncrit"],
                                              precision=case["precision"]))
    x, q, w = _inputs(case, seed)
    st = dict(case=case, x=x, q=q, w=w)
    if kind == "step":
        st["f"] = _handle(case)
        if case["host"]:
            st["x"], st["q"] = x.cpu().numpy(), q.cpu().numpy()
    elif kind == "matvec":
        # the tree is built with other charges than the product uses
        st["f"] = _handle(case).build(x, torch.ones_like(q))
        st["phi"], st["grad"] = torch.empty_like(q), torch.empty_like(x)
    elif kind == "energy":
        for k in ("x", "q", "w"):
            st[k].requires_grad_()
    elif kind == "sort":
        st["keys"] = torch.empty(case["n"], dtype=torch.int64, device="cuda")
        st["perm"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "step":
        return st["f"].build(st["x"], st["q"]).evaluate()
    if kind == "matvec":
        st["f"].update_charges(st["q"])
        return st["f"].evaluate(st["phi"], st["grad"])
    if kind == "energy":
        e = fmm_energy(st["x"], st["q"], st["w"], p=case["p"], theta=case["theta"], ncrit=case["ncrit"],
                       precision=case["precision"])
        return (e.detach(),) + torch.autograd.grad(e, (st["x"], st["q"], st["w"]))
    if kind == "batch":
        return [t for pair in st["batch"].evaluate() for t in pair]
    rc = lib().fmm_morton_sort_noalloc(ctypes.c_void_p(st["x"].data_ptr()), case["n"],
                                       FMM_F64 if case["dtype"] == "f64" else FMM_F32,
                                       ctypes.c_void_p(st["keys"].data_ptr()), ctypes.c_void_p(st["perm"].data_ptr()),
                                       ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if rc != 0:
        raise RuntimeError("fmm_morton_sort_noalloc: %d" % rc)
    return st["keys"], st["perm"]


# -- what a pass cannot do without ---------------------------------------------

def _fmm_flops(n, p, theta, ncrit):
    """Near field (20 flop per interaction) and same-level translations (2 p^4
    flop each) of an octree over n particles of a uniform cube, whose leaves are
    the first full level with at most ncrit particles per cell on average; an
    estimate for the clustered trees."""
    depth = 0
    while n / 8.0 ** depth > ncrit * 0.8:
        depth += 1
    r = math.ceil(2 * math.sqrt(3) / theta) + 1
    near = [(a, b, c) for a in range(-r, r + 1) for b in range(-r, r + 1) for c in range(-r, r + 1)
            if 3.0 >= theta * theta * (a * a + b * b + c * c)]

    def pairs(level):
        s = 2 ** level
        return sum((s - abs(a)) * (s - abs(b)) * (s - abs(c)) for a, b, c in near
                   if max(abs(a), abs(b), abs(c)) < s)

    m2l = sum(64 * pairs(level - 1) - pairs(level) for level in range(1, depth + 1))
    return 20.0 * pairs(depth) * (n / 8.0 ** depth) ** 2 + 2.0 * p ** 4 * m2l


def work(case):
    n, size = case["n"], 8 if case["dtype"] == "f64" else 4
    if case["kind"] == "sort":
        return {"bytes": n * (3 * size + 12), "flops": 0}
    args = case["p"], case["theta"], case["ncrit"]
    if case["kind"] == "batch":
        sizes = _sizes(case, 0)
        return {"bytes": 8 * size * sum(sizes), "flops": sum(_fmm_flops(m, *args) for m in sizes)}
    flops = _fmm_flops(n, *args)
    if case["kind"] == "matvec":
        return {"bytes": n * 5 * size, "flops": flops}
    if case["kind"] == "energy":
        return {"bytes": n * 10 * size, "flops": 2 * flops}
    return {"bytes": n * 8 * size, "flops": flops}


# -- what a result may differ by -------------------------------------------------

def tolerance(case):
    if case["kind"] == "sort":
        return "exact"
    if case["precision"] == "fp64":
        return {"rel": 1e-14}  # the two translation engines (rotated, dense) differ by up to 7e-16, their near field being the same
    if case["kind"] == "energy":
        return {"rel": 7e-6}  # the energy itself, a sum of both signs, is 1.7e-6 from the FP64 path's
    return {"rel": 5e-6}  # mixed and FP64 results on one tree differ by up to 1.2e-6 over these ranges


def _direct(x, q):
    """Potential and gradient by direct summation in FP64."""
    x, q = x.double(), q.double()
    n = x.shape[0]
    step = max(1, 200000000 // n)
    phi, grad = torch.empty_like(q), torch.empty_like(x)
    for a in range(0, n, step):
        t = x[a:a + step]
        d = [x[:, k][None, :] - t[:, k][:, None] for k in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        inv = torch.where(r2 > 0, r2.rsqrt(), 0.0)
        s = inv * q[None, :]
        phi[a:a + step] = s.sum(1)
        s = s * inv * inv
        for k in range(3):
            grad[a:a + step, k] = (s * d[k]).sum(1)
    return phi, grad


def exact(case, seed):
    """The direct sum the method approximates, in FP64 (the method's own
    truncation, set by p and theta, is part of the distance to it)."""
    kind, n = case["kind"], case["n"]
    if kind == "batch":
        if sum(float(m) * m for m in _sizes(case, seed)) > EXACT_MAX_PAIRS:
            return None
        return [t for x, q in _inputs(case, seed) for t in _direct(x, q)]
    if kind != "sort" and float(n) * n * (2 if kind == "energy" else 1) > EXACT_MAX_PAIRS:
        return None
    x, q, w = _inputs(case, seed)
    if kind == "sort":
        return _exact_sort(x)
    phi, grad = _direct(x, q)
    if kind != "energy":
        return (phi.cpu().numpy(), grad.cpu().numpy()) if case["host"] else (phi, grad)
    q, w = q.double(), w.double()
    psi, gpsi = _direct(x, w * q)
    return (0.5 * (w * q * phi).sum(), 0.5 * q[:, None] * (w[:, None] * grad + gpsi), 0.5 * (w * phi + psi), 0.5 * q * phi)


def _exact_sort(x):
    x = x.double()
    lo, hi = x.min(0).values, x.max(0).values
    half = ((hi - lo) / 2).max()
    half = torch.where(half > 0, half, torch.ones_like(half))
    i = (x - ((lo + hi) / 2 - half)) * (2.0 ** 21 / (2 * half))
    i = i.floor().clamp(0, 2 ** 21 - 1).long()
    key = torch.zeros_like(i[:, 0])
    for b in range(21):
        for k in range(3):
            key |= ((i[:, k] >> b) & 1) << (3 * b + k)
    key, perm = torch.sort(key, stable=True)
    return key, perm.int()
