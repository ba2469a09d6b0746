"""The workloads whose speed is measured, through the package's public calls.

A case is a dict of plain values.  ``kind`` says which call a program makes:

  apply    sweeps of one local function over one grid (builtin or run-time
           compiled source; forward Euler or SSP-RK3): ``apply``
  batch    many uneven 2D grids advanced together: ``apply_batch``
  adjoint  loss and gradients of a diffusion run by the discrete adjoint with
           checkpointed recomputation: ``adjoint``

``shape`` is written "slow x ... x fast", ``bc`` one letter per axis in the same
order (p periodic, d Dirichlet 0).  Sizes come from the benchmark's workloads
and the test suite; ``draw`` spreads over the ranges between them.
"""
from __future__ import annotations

import functools
import random

import torch

import paper_1502_03504_gb300 as L

_DT = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
_ESIZE = {"f64": 8, "f32": 4, "bf16": 2}

# Builtins: parameters, declared halo, fields, floating-point operations per
# point and sweep (adds, multiplies and FMAs counted as 1, 1 and 2).
_BUILTIN = {
    "jacobi5": ([0.2], 1, 1, 7),
    "star9r2": ([0.1], 2, 1, 13),
    "diff7": ([0.1], 1, 1, 9),
    "swe_cgrid": ([0.02, 1.0, 1.0], 1, 3, 11),
    "swe_flux": ([0.02, 1.0, 0.5, 1.0], 1, 3, 52),
}
# Gray-Scott reaction-diffusion, written as a user writes a local function.
_GRAY_SCOTT = """
const C u = U(0, 0, 0), v = U(1, 0, 0);
const C lu = fma_(C(-4), u, add(add(U(0, -1, 0), U(0, 1, 0)), add(U(0, 0, -1), U(0, 0, 1))));
const C lv = fma_(C(-4), v, add(add(U(1, -1, 0), U(1, 1, 0)), add(U(1, 0, -1), U(1, 0, 1))));
const C uvv = mul(u, mul(v, v));
out[0] = fma_(P[0], fma_(P[1], lu, fma_(P[3], sub(C(1), u), -uvv)), u);
out[1] = fma_(P[0], fma_(P[2], lv, fma_(-add(P[3], P[4]), v, uvv)), v);
"""
_GS_PRM = [1.0, 0.16, 0.08, 0.035, 0.065]
_GS_FLOPS = 31


def listed():
    return [
        # the smallest call: a small ragged plate, where latency and launches count
        dict(name="plate_100x200_f32", kind="apply", fn="jacobi5", dtype="f32", shape="100x200",
             bc="dd", steps=20, scheme="euler"),
        # double-precision heat equation on a grid that stays in L2
        dict(name="heat_256_f64", kind="apply", fn="jacobi5", dtype="f64", shape="256x256",
             bc="pp", steps=100, scheme="euler"),
        # 2D heat equation whose row pitch is no multiple of 16 bytes
        dict(name="heat_7094_f32", kind="apply", fn="jacobi5", dtype="f32", shape="7094x7094",
             bc="pd", steps=20, scheme="euler"),
        # fourth-order 2D diffusion at scale
        dict(name="star9r2_8192_f32", kind="apply", fn="star9r2", dtype="f32", shape="8192x8192",
             bc="pp", steps=50, scheme="euler"),
        # 3D diffusion at scale: the headline grid
        dict(name="diff7_512_f32", kind="apply", fn="diff7", dtype="f32", shape="512x512x512",
             bc="ddd", steps=50, scheme="euler"),
        # 3D diffusion on a ragged channel: rows of any pitch, one periodic axis
        dict(name="diff7_130x500x510_f32", kind="apply", fn="diff7", dtype="f32",
             shape="130x500x510", bc="dpd", steps=20, scheme="euler"),
        # linearised shallow water, three coupled fields, full and reduced storage
        dict(name="swe_4096_f32", kind="apply", fn="swe_cgrid", dtype="f32", shape="4096x4096",
             bc="pp", steps=200, scheme="euler"),
        dict(name="swe_4096_bf16", kind="apply", fn="swe_cgrid", dtype="bf16", shape="4096x4096",
             bc="pp", steps=200, scheme="euler"),
        # nonlinear shallow water (corner taps) under a three-stage time scheme
        dict(name="swe_flux_rk3_4096_f32", kind="apply", fn="swe_flux", dtype="f32",
             shape="4096x4096", bc="pp", steps=50, scheme="rk3"),
        # a user's own two-field nonlinear local function, compiled at run time
        dict(name="gray_scott_4096_f32", kind="apply", fn="gray_scott", dtype="f32",
             shape="4096x4096", bc="pp", steps=100, scheme="euler"),
        # an ensemble of uneven 2D grids in one call
        dict(name="batch_512_f32", kind="batch", fn="jacobi5", dtype="f32", grids=512, lo=64,
             hi=2048, shapes_seed=1003, steps=20),
        # training step: forward, loss and both gradients of a 3D diffusion
        dict(name="adjoint_256_f32", kind="adjoint", fn="diff7", dtype="f32", shape="256x256x256",
             bc="ppp", steps=100, ckpt=10),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    import math

    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _side(rng, lo, hi):
    """A side, log-uniform; one in two a multiple of 8 as programs like them."""
    n = _log_int(rng, lo, hi)
    return max(lo, n // 8 * 8) if rng.random() < 0.5 else n


def draw(rng):
    """One more case of the same ranges, no dearer than the largest listed one."""
    what = rng.choice(["plane", "plane", "volume", "volume", "shallow", "shallow", "source", "batch",
                       "adjoint"])
    bc2 = rng.choice(["pp", "dd", "pd", "dp"])
    bc3 = rng.choice(["ppp", "ddd", "ddd", "dpd", "pdd"])
    if what == "plane":
        shape = "%dx%d" % (_side(rng, 100, 8192), _side(rng, 100, 8192))
        dtype = rng.choice(["f32", "f32", "bf16", "f64"])
        cap = 3.3e9 if dtype != "f64" else 4e8
        return dict(kind="apply", fn=rng.choice(["jacobi5", "star9r2"]), dtype=dtype, shape=shape,
                    bc=bc2, steps=_steps(rng, shape, cap), scheme="euler")
    if what == "volume":
        shape = "x".join(str(_side(rng, 40, 512)) for _ in range(3))
        dtype = rng.choice(["f32", "f32", "f32", "bf16", "f64"])
        cap = 6e9 if dtype != "f64" else 4e8
        return dict(kind="apply", fn="diff7", dtype=dtype, shape=shape, bc=bc3,
                    steps=_steps(rng, shape, cap), scheme="euler")
    if what == "shallow":
        shape = "%dx%d" % (_side(rng, 100, 4096), _side(rng, 100, 4096))
        fn, scheme = rng.choice([("swe_cgrid", "euler"), ("swe_flux", "euler"), ("swe_flux", "rk3")])
        cap = 3e9 if scheme == "euler" else 8e8
        return dict(kind="apply", fn=fn, dtype=rng.choice(["f32", "bf16"]), shape=shape, bc=bc2,
                    steps=_steps(rng, shape, cap), scheme=scheme)
    if what == "source":
        shape = "%dx%d" % (_side(rng, 100, 4096), _side(rng, 100, 4096))
        return dict(kind="apply", fn="gray_scott", dtype="f32", shape=shape, bc=bc2,
                    steps=_steps(rng, shape, 1.6e9), scheme="euler")
    if what == "batch":
        return dict(kind="batch", fn=rng.choice(["jacobi5", "star9r2"]), dtype="f32",
                    grids=_log_int(rng, 16, 512), lo=64, hi=_log_int(rng, 200, 2048),
                    shapes_seed=rng.randrange(1 << 20), steps=_log_int(rng, 4, 20))
    if rng.random() < 0.5:
        shape = "x".join(str(_side(rng, 40, 256)) for _ in range(3))
        return dict(kind="adjoint", fn="diff7", dtype="f32", shape=shape,
                    bc=rng.choice(["ppp", "ddd"]), steps=_steps(rng, shape, 1.6e9), ckpt=10)
    shape = "%dx%d" % (_side(rng, 100, 2048), _side(rng, 100, 2048))
    return dict(kind="adjoint", fn="jacobi5", dtype="f32", shape=shape, bc=rng.choice(["pp", "dd"]),
                steps=_steps(rng, shape, 4e8), ckpt=10)


def _steps(rng, shape, cap):
    pts = 1
    for n in _shape(shape):
        pts *= n
    return _log_int(rng, 1, max(1, min(200, int(cap / pts))))


def _shape(text):
    return tuple(int(n) for n in text.split("x"))


def _bc(letters):
    return [L.BC_PERIODIC if b == "p" else L.BC_DIRICHLET for b in letters]


def _fields(case, shape, seed, device):
    """The initial state: a user's arrays, made from the seed alone."""
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    rand = lambda: torch.rand(shape, generator=g, device=device, dtype=torch.float32)  # noqa: E731
    randn = lambda: torch.randn(shape, generator=g, device=device, dtype=torch.float32)  # noqa: E731
    if case["fn"].startswith("swe"):
        # swe_cgrid in full storage holds h = 1 + eta; BF16 and swe_flux hold eta
        h = 0.01 * randn()
        if case["fn"] == "swe_cgrid" and case["dtype"] != "bf16":
            h = h + 1.0
        x = [h, 0.1 * randn(), 0.1 * randn()]
    elif case["fn"] == "gray_scott":
        x = [1.0 - 0.3 * rand(), 0.25 * rand()]
    else:
        x = [rand()]
    return [t.to(_DT[case["dtype"]]) for t in x]


@functools.lru_cache(maxsize=None)
def _source(dtype):
    # a program compiles its local function once
    return L.Stencil.source(_GRAY_SCOTT, ndim=2, radius=1, nfields=2, params=_GS_PRM).compile(dtype)


@functools.lru_cache(maxsize=None)
def _workspace(nbytes):
    # a program keeps one workspace per problem size for its life; its calls
    # follow one another on one stream
    return torch.empty(nbytes, dtype=torch.uint8, device="cuda")


def _stencil(case):
    if case["fn"] == "gray_scott":
        return _source(case["dtype"]), 1, 2
    prm, halo, nf, _ = _BUILTIN[case["fn"]]
    st = L.Stencil.builtin(case["fn"], *prm)
    if case.get("scheme", "euler") != "euler":
        st.set_scheme(case["scheme"])
    return st, halo, nf


def _batch_shapes(case):
    """Sides U{lo..hi} and one boundary kind per grid, from the case alone."""
    rng = random.Random(case["shapes_seed"])
    out = []
    for _ in range(case["grids"]):
        ny, nx = rng.randint(case["lo"], case["hi"]), rng.randint(case["lo"], case["hi"])
        out.append((ny, nx, "pp" if rng.random() < 0.5 else "dd"))
    return out


def _pool(case):
    """Offsets of the batch's grids in one pool (each on a 256-byte boundary)."""
    offs, n = [], 0
    for ny, nx, _ in _batch_shapes(case):
        offs.append(n)
        n += (ny * nx + 63) // 64 * 64
    return offs, n


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "batch":
        shapes, (offs, n) = _batch_shapes(case), _pool(case)
        st, halo, _ = _stencil(case)
        u = _fields(case, (n,), seed, dev)[0]
        o, w = torch.zeros_like(u), torch.zeros_like(u)
        view = lambda t: [t[a:a + ny * nx].view(ny, nx) for a, (ny, nx, _) in zip(offs, shapes)]  # noqa: E731
        grids = []
        for ny, nx, bc in shapes:
            grids.append(L.Grid((ny, nx), case["dtype"], halo=halo).set_boundaries(_bc(bc)))
        ws = _workspace(L.batch_workspace_size(grids, st))
        return dict(kind="batch", grids=grids, st=st, ins=view(u), outs=view(o), works=view(w),
                    ws=ws, pool=o, steps=case["steps"])
    shape = _shape(case["shape"])
    st, halo, nf = _stencil(case)
    g = L.Grid(shape, case["dtype"], halo=halo, nfields=nf).set_boundaries(_bc(case["bc"]))
    ins = _fields(case, shape, seed, dev)
    if case["kind"] == "adjoint":
        gen = torch.Generator(device=dev)
        gen.manual_seed(int(seed) + 7919)
        target = torch.randn(shape, generator=gen, device=dev).to(_DT[case["dtype"]])
        ws = _workspace(L.workspace_size(g, st, case["steps"], case["ckpt"]))
        return dict(kind="adjoint", g=g, st=st, u0=ins[0], target=target, grad=torch.empty_like(ins[0]),
                    ws=ws, steps=case["steps"], ckpt=case["ckpt"])
    outs = [torch.empty_like(t) for t in ins]
    ns = st.work_states()
    works = [torch.empty((ns,) + shape, dtype=t.dtype, device=dev) for t in ins]
    return dict(kind="apply", g=g, st=st, ins=ins, outs=outs, works=works, steps=case["steps"])


def run(state):
    s = state
    if s["kind"] == "batch":
        L.apply_batch(s["grids"], s["st"], s["ins"], s["outs"], s["works"], nsteps=s["steps"],
                      workspace=s["ws"])
        return s["pool"]
    if s["kind"] == "adjoint":
        loss, grad, gc = L.adjoint(s["g"], s["st"], s["u0"], s["target"], s["steps"], s["ckpt"],
                                   grad_u0=s["grad"], workspace=s["ws"])
        return {"loss": loss, "grad_u0": grad, "grad_c": gc}
    return L.apply(s["g"], s["st"], s["ins"], out=s["outs"], work=s["works"], nsteps=s["steps"])


def work(case):
    esz = _ESIZE[case["dtype"]]
    if case["kind"] == "batch":
        pts = sum(ny * nx for ny, nx, _ in _batch_shapes(case))
        return {"bytes": 2 * esz * pts, "flops": _BUILTIN[case["fn"]][3] * pts * case["steps"]}
    pts = 1
    for n in _shape(case["shape"]):
        pts *= n
    if case["kind"] == "adjoint":
        # reads u0 and the target, writes dL/du0; forward sweeps, transposed
        # sweeps with one FMA per point for dL/dc
        f = _BUILTIN[case["fn"]][3]
        return {"bytes": 3 * esz * pts, "flops": (2 * f + 2) * pts * case["steps"]}
    f, nf = (_GS_FLOPS, 2) if case["fn"] == "gray_scott" else (_BUILTIN[case["fn"]][3],
                                                               _BUILTIN[case["fn"]][2])
    stages = 3 if case["scheme"] == "rk3" else 1
    per = f * stages + (3 * nf * (stages - 1))
    return {"bytes": 2 * esz * nf * pts, "flops": per * pts * case["steps"]}


# ------------------------------------------------------------------ 64-bit values
def _ghosted(u, bc, r):
    """u with r ghost cells per side: wrapped (p) or 0 (d); the slowest axis last, so it decides."""
    for ax in range(u.dim() - 1, -1, -1):
        n = u.shape[ax]
        if bc[ax] == "p":
            idx = torch.arange(-r, n + r, device=u.device) % n
            u = u.index_select(ax, idx)
        else:
            pad = [0] * (2 * u.dim())
            pad[2 * (u.dim() - 1 - ax)] = pad[2 * (u.dim() - 1 - ax) + 1] = r
            u = torch.nn.functional.pad(u, pad)
    return u


def _tap(p, shape, r, *offs):
    """The ghosted field p at offsets (slowest axis first)."""
    return p[tuple(slice(r + o, r + o + n) for o, n in zip(offs, shape))]


def _laplacian(fn, u, bc):
    r = 2 if fn == "star9r2" else 1
    p, s, d = _ghosted(u, bc, r), u.shape, u.dim()
    unit = [tuple(k if a == ax else 0 for a in range(d)) for ax in range(d) for k in (-1, 1)]
    near = sum(_tap(p, s, r, *o) for o in unit)
    if fn == "star9r2":
        far = sum(_tap(p, s, r, *(2 * k for k in o)) for o in unit)
        return (4.0 / 3.0) * near - far / 12.0 - 5.0 * u
    return near - 2.0 * d * u


def _euler(fn, x, bc):
    if fn in ("jacobi5", "star9r2", "diff7"):
        return [x[0] + _BUILTIN[fn][0][0] * _laplacian(fn, x[0], bc)]
    if fn == "gray_scott":
        dt, du, dv, f, k = _GS_PRM
        u, v = x
        uvv = u * v * v
        return [u + dt * (du * _laplacian("jacobi5", u, bc) + f * (1.0 - u) - uvv),
                v + dt * (dv * _laplacian("jacobi5", v, bc) - (f + k) * v + uvv)]
    s = x[0].shape
    P = [_ghosted(t, bc, 1) for t in x]
    U = lambda f, dx, dy: _tap(P[f], s, 1, dy, dx)  # noqa: E731
    e, u, v = x
    if fn == "swe_cgrid":
        dt, g, H = _BUILTIN[fn][0]
        return [e - dt * H * (u - U(1, -1, 0) + v - U(2, 0, -1)),
                u - dt * g * (U(0, 1, 0) - e), v - dt * g * (U(0, 0, 1) - e)]
    dt, g, f, H = _BUILTIN[fn][0]
    dF = (H + 0.5 * (e + U(0, 1, 0))) * u - (H + 0.5 * (U(0, -1, 0) + e)) * U(1, -1, 0)
    dG = (H + 0.5 * (e + U(0, 0, 1))) * v - (H + 0.5 * (U(0, 0, -1) + e)) * U(2, 0, -1)
    vb = 0.25 * (v + U(2, 1, 0) + U(2, 0, -1) + U(2, 1, -1))
    ub = 0.25 * (u + U(1, -1, 0) + U(1, 0, 1) + U(1, -1, 1))
    au = -0.5 * (u * (U(1, 1, 0) - U(1, -1, 0)) + vb * (U(1, 0, 1) - U(1, 0, -1)))
    av = -0.5 * (ub * (U(2, 1, 0) - U(2, -1, 0)) + v * (U(2, 0, 1) - U(2, 0, -1)))
    return [e - dt * (dF + dG), u + dt * (f * vb - g * (U(0, 1, 0) - e) + au),
            v + dt * (-f * ub - g * (U(0, 0, 1) - e) + av)]


def _advance(fn, x, bc, steps, scheme):
    for _ in range(steps):
        e = _euler(fn, x, bc)
        if scheme == "rk3":
            e = [0.75 * a + 0.25 * b for a, b in zip(x, _euler(fn, e, bc))]
            e = [a / 3.0 + 2.0 / 3.0 * b for a, b in zip(x, _euler(fn, e, bc))]
        x = e
    return x


def exact(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "batch":
        shapes, (offs, n) = _batch_shapes(case), _pool(case)
        u = _fields(case, (n,), seed, dev)[0]
        out = torch.zeros(n, dtype=torch.float64, device=dev)
        for a, (ny, nx, bc) in zip(offs, shapes):
            x = u[a:a + ny * nx].view(ny, nx).double()
            out[a:a + ny * nx] = _advance(case["fn"], [x], bc, case["steps"], "euler")[0].reshape(-1)
        return out
    shape = _shape(case["shape"])
    x = [t.double() for t in _fields(case, shape, seed, dev)]
    if case["kind"] == "apply":
        return _advance(case["fn"], x, case["bc"], case["steps"], case["scheme"])
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) + 7919)
    target = torch.randn(shape, generator=gen, device=dev).to(_DT[case["dtype"]]).double()
    # u' = u + c L u, and L is its own transpose on these boundaries: dL/du0 is
    # lambda swept back, dL/dc the sum of <lambda_{t+1}, L u_t>
    states = [x[0]]
    for _ in range(case["steps"]):
        states.append(_euler(case["fn"], [states[-1]], case["bc"])[0])
    lam = 2.0 * (states[-1] - target)
    loss = (states[-1] - target).square().sum()
    gc = torch.zeros((), dtype=torch.float64, device=dev)
    for t in range(case["steps"] - 1, -1, -1):
        gc += (lam * _laplacian(case["fn"], states[t], case["bc"])).sum()
        lam = _euler(case["fn"], [lam], case["bc"])[0]
    return {"loss": float(loss), "grad_u0": lam, "grad_c": float(gc)}
