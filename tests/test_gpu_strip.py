"""Register strips (path 5): K sweeps of a 2D function per launch with every
intermediate state in registers.

Every sweep rounds to the storage precision, so the result must equal one
sweep per launch on the direct kernel bitwise: at the edges of the strips (the
valid width is 120 or 112 columns), of the chunks and of the grid, for rows of
any pitch, periodic and Dirichlet sides with zero and non-zero values, every
depth, odd sweep counts, box and star functions, several fields, both
multi-stage schemes and run-time compiled functions.
"""
import numpy as np
import pytest
import torch

import lope_inputs as LI
from gpu_helpers import to_device
from user_bodies import GRAY_SCOTT

pytestmark = pytest.mark.gpu

DIRECT, STRIP = 3, 5
BCS = [([0, 0], None), ([1, 1], None), ([0, 1], [0.0, (0.5, -0.25)]), ([(1, 1), 0], [(0.3, 0.7), 0.0]),
       ([1, 1], [(0.3, -0.2), (0.0, 0.5)])]
FUNCS = {
    "jacobi5": ([0.2], 1, 1, (8, 4, 2, 1)),
    "star9r2": ([0.1], 2, 1, (4, 2, 1)),
    "swe_cgrid": ([0.02, 1.0, 1.0], 1, 3, (6, 4, 2, 1)),
    "swe_flux": ([0.02, 1.0, 0.5, 1.0], 1, 3, (4, 2, 1)),
}


def _run(L, g, st, f, T, launch):
    o = L.apply(g, st, f, nsteps=T, launch=launch)
    torch.cuda.synchronize()
    L.sync_status()
    return o


def _fields(shape, dtype, nf, seed):
    x = LI.swe_fields(seed, shape) if nf == 3 else [LI.uniform_field(seed, shape, k * 10 ** 6) for k in range(nf)]
    return [to_device(a - 1.0 if nf == 3 and k == 0 else a, dtype)[0] for k, a in enumerate(x)]


def _check(L, g, st, f, T, k):
    ref = _run(L, g, st, f, T, L.Launch(DIRECT, 0, 0, 0, -1))
    got = _run(L, g, st, f, T, L.Launch(STRIP, 0, 0, k, -1))
    for a, b in zip(got, ref):
        assert torch.equal(a, b), (g.shape, T, k)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("name", list(FUNCS))
@pytest.mark.parametrize("shape", [(40, 4), (3, 120), (65, 124), (200, 112), (1030, 232), (17, 1000)],
                         ids=lambda s: "x".join(map(str, s)))
def test_strips_bitwise_equal_direct(lope, name, shape, dtype):
    prm, halo, nf, depths = FUNCS[name]
    st = lope.Stencil.builtin(name, *prm)
    f = _fields(shape, dtype, nf, 1800)
    for bc, bv in BCS:
        g = lope.Grid(shape, dtype, halo=halo, nfields=nf).set_boundaries(bc, bv)
        for k in depths:
            _check(lope, g, st, f, k, k)
    _check(lope, g, st, f, 2 * depths[0] + 3, depths[0])  # passes of several depths


@pytest.mark.parametrize("name", list(FUNCS))
@pytest.mark.parametrize("shape", [(5, 1), (9, 3), (65, 119), (130, 225), (70, 1001)],
                         ids=lambda s: "x".join(map(str, s)))
def test_strips_rows_of_any_pitch(lope, name, shape):
    prm, halo, nf, depths = FUNCS[name]
    st = lope.Stencil.builtin(name, *prm)
    f = _fields(shape, "f32", nf, 1810)
    for bc, bv in BCS:
        if halo > 1 and shape[1] < halo and bc[1] == 0:
            continue  # a periodic axis shorter than the radius is refused
        g = lope.Grid(shape, "f32", halo=halo, nfields=nf).set_boundaries(bc, bv)
        for k in depths:
            _check(lope, g, st, f, k, k)


def test_strips_weight_tables(lope):
    rng = np.random.default_rng(1820)
    shape = (90, 236)
    for r in (1, 2):
        w = rng.uniform(0.0, 0.08, (2 * r + 1, 2 * r + 1))
        w[r, r] = 1.0 - (w.sum() - w[r, r])
        star = np.zeros_like(w)
        star[r], star[:, r] = w[r], w[:, r]
        for table in (w, star):
            st = lope.Stencil.linear(table)
            for dtype in ("f32", "bf16"):
                f = _fields(shape, dtype, 1, 1821)
                for bc, bv in BCS:
                    g = lope.Grid(shape, dtype, halo=r).set_boundaries(bc, bv)
                    _check(lope, g, st, f, 7, 4)


@pytest.mark.parametrize("scheme", ["rk2", "rk3"])
@pytest.mark.parametrize("name", list(FUNCS))
def test_strips_multi_stage(lope, name, scheme):
    prm, halo, nf, _ = FUNCS[name]
    st = lope.Stencil.builtin(name, *prm).set_scheme(scheme)
    for shape in ((77, 124), (300, 232)):
        for dtype in ("f32", "bf16"):
            f = _fields(shape, dtype, nf, 1830)
            for bc, bv in BCS:
                g = lope.Grid(shape, dtype, halo=halo, nfields=nf).set_boundaries(bc, bv)
                _check(lope, g, st, f, 3, 1)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_strips_run_time_compiled(lope, dtype):
    prm = [1.0, 0.16, 0.08, 0.035, 0.065]
    st = lope.Stencil.source(GRAY_SCOTT, ndim=2, radius=1, nfields=2, params=prm)
    for shape in ((61, 124), (200, 360)):
        f = _fields(shape, dtype, 2, 1840)
        for bc, bv in BCS:
            g = lope.Grid(shape, dtype, halo=1, nfields=2).set_boundaries(bc, bv)
            for T, k in ((4, 4), (7, 4), (3, 2)):
                _check(lope, g, st, f, T, k)


# A function of NF fields and radius R whose every tap is checked: a value
# outside [0.9, 2.1] sets the device error flag.  Its result is a mean, so states
# and boundary values in [1, 2] stay there.  (C is float or a pair of floats.)
CHECKED = """
bool good = true;
auto seen = [&](C v) {
  const float* w = reinterpret_cast<const float*>(&v);
  for (int i = 0; i < int(sizeof(C) / 4); ++i) good &= w[i] >= 0.9f && w[i] <= 2.1f;
  return v;
};
for (int f = 0; f < NF; ++f) {
  C s = seen(U((f + 1) % NF, 0, 0));
  for (int k = 1; k <= R; ++k) {
    s = add(s, add(seen(U(f, -k, 0)), seen(U(f, k, 0))));
    s = add(s, add(seen(U(f, 0, -k)), seen(U(f, 0, k))));
  }
  out[f] = mul(P[0], s);
}
if (!good) raise_error(err, 2);
"""


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("nf,radius", [(1, 1), (2, 1), (3, 1), (1, 2), (2, 2), (3, 2)])
def test_strips_show_a_function_only_states_and_boundary_values(lope, dtype, nf, radius):
    """A run-time compiled function of every shape, whatever rows its pipeline
    fills or drains: no tap is anything but a state or a boundary value, and the
    result is the direct kernel's."""
    st = lope.Stencil.source(CHECKED, ndim=2, radius=radius, nfields=nf, params=[1.0 / (4 * radius + 1)])
    for shape in ((2, 4), (3, 124), (40, 116), (67, 360), (513, 128)):
        f = [1.0 + t for t in _fields(shape, dtype, 1, 1880)] * nf
        f = [t.clone() for t in f]
        for bc in ([0, 0], [1, 1], [1, 0]):
            g = lope.Grid(shape, dtype, halo=radius, nfields=nf).set_boundaries(bc, [1.5 if b else 0.0 for b in bc])
            for T, k in ((4, 4), (2, 2), (1, 1), (7, 4)):
                _check(lope, g, st, f if nf > 1 else f[0:1], T, k)


def test_strips_computed_taps(lope):
    """Offsets computed at run time: inside the halo as on the direct kernel;
    beyond it clamped and reported."""
    g = lope.Grid((64, 128), "f32", halo=1)
    u = torch.rand(64, 128, device="cuda")
    body = "C s = C(0);\nfor (int d = -1; d <= %d; ++d) s = add(s, add(U(0, d, 0), U(0, 0, d)));\nout[0] = s;"
    inside = lope.Stencil.source(body % 1, ndim=2, radius=1)
    _check(lope, g, inside, [u], 7, 4)
    beyond = lope.Stencil.source(body % 2, ndim=2, radius=1)
    lope.apply(g, beyond, u, nsteps=4, launch=lope.Launch(STRIP, 0, 0, 4, -1))
    with pytest.raises(lope.LopeError, match="outside its declared halo"):
        lope.sync_status()
    _check(lope, g, inside, [u], 4, 4)


def test_strips_default_plan_and_refusals(lope):
    """Twelve sweeps or more take the strips; what they cannot run is refused."""
    shape = (64, 132)
    u = torch.rand(shape, device="cuda")
    o, w = torch.empty_like(u), torch.empty_like(u)
    st = lope.Stencil.builtin("jacobi5", 0.2)
    g = lope.Grid(shape, "f32", halo=1)
    plan, n = lope.plan(g, st, u, o, w, nsteps=23)
    assert (plan.path, plan.tsteps, n) == (STRIP, 8, 5)  # 8 + 8 + 4 + 2 + 1
    assert lope.plan(g, st, u, o, w, nsteps=11)[0].path != STRIP
    ref = _run(lope, g, st, u, 23, lope.Launch(DIRECT, 0, 0, 0, -1))
    assert torch.equal(_run(lope, g, st, u, 23, None), ref)
    for bad in (3, 6, 16):
        with pytest.raises(lope.LopeError, match="UNSUPPORTED"):
            lope.apply(g, st, u, nsteps=23, launch=lope.Launch(STRIP, 0, 0, bad, -1))
    d = torch.rand(shape, device="cuda", dtype=torch.float64)
    with pytest.raises(lope.LopeError, match="UNSUPPORTED"):
        lope.apply(lope.Grid(shape, "f64", halo=1), st, d, nsteps=4, launch=lope.Launch(STRIP, 0, 0, 4, -1))


@pytest.mark.parametrize("shape", [(1, 1), (8, 32), (100, 300), (257, 255), (530, 515)],
                         ids=lambda s: "x".join(map(str, s)))
def test_double_default_plan_equals_direct(lope, shape):
    """The FP64 tile and depth depend on the grid's size: the default plan's
    result against one sweep per launch, also where the sweeps leave a rest."""
    f = [to_device(LI.uniform_field(1840, shape, 0), "f64")[0]]
    box = np.random.default_rng(5).uniform(-0.1, 0.1, (5, 5))
    for st, halo in [(lope.Stencil.builtin("jacobi5", 0.2), 1), (lope.Stencil.builtin("star9r2", 0.1), 2),
                     (lope.Stencil.linear(box), 2)]:
        for bc, bv in BCS[:3]:
            if bc[0] == 0 and min(shape) < halo:
                continue
            g = lope.Grid(shape, "f64", halo=halo).set_boundaries(bc, bv)
            ref = _run(lope, g, st, f, 15, lope.Launch(DIRECT, 0, 0, 0, -1))
            got = _run(lope, g, st, f, 15, None)
            assert torch.equal(got[0], ref[0]), (shape, halo, bc)


@pytest.mark.parametrize("shape", [(300, 200), (97, 203)], ids=lambda s: "x".join(map(str, s)))
def test_strips_write_only_their_output(lope, shape):
    n = int(np.prod(shape))
    guard, sentinel = 4096, -7.0e30
    u = torch.rand(shape, device="cuda")
    keep = u.clone()
    st = lope.Stencil.builtin("jacobi5", 0.2)
    for bc in ([0, 0], [1, 1]):
        g = lope.Grid(shape, "f32", halo=1).set_boundaries(bc)
        bufs = [torch.full((n + 2 * guard,), sentinel, device="cuda") for _ in range(2)]
        out, work = (b[guard:guard + n].view(shape) for b in bufs)
        lope.apply(g, st, u, out=out, work=work, nsteps=13, launch=lope.Launch(STRIP, 0, 0, 8, -1))
        torch.cuda.synchronize()
        for b in bufs:
            assert bool((b[:guard] == sentinel).all()) and bool((b[guard + n:] == sentinel).all())
        assert torch.equal(u, keep)


@pytest.mark.parametrize("kind,prm,halo,depths", [("jacobi5", [0.2], 1, (8, 4, 2, 1)),
                                                  ("star9r2", [0.1], 2, (4, 2, 1))])
def test_batched_strips_equal_each_grid_alone(lope, kind, prm, halo, depths):
    """Uneven grids of aligned and odd widths (fewer columns than a lane's,
    one strip, several), both boundary kinds, every depth and a sweep count
    that takes passes of each; then again in memory freed and allocated anew."""
    shapes = [(1, 7), (130, 3), (40, 4), (65, 113), (200, 224), (17, 500), (300, 251), (90, 120)]
    st = lope.Stencil.builtin(kind, *prm)

    def once(T, launch):
        grids, ins = [], []
        for i, s in enumerate(shapes):
            g = lope.Grid(s, "f32", halo=halo)
            if i % 2 == 0:
                g.set_boundaries([(1, 1), (1, 1)], [(0.3, -0.2), (0.0, 0.5)])
            grids.append(g)
            ins.append(to_device(LI.uniform_field(1850 + i, s), "f32")[0])
        outs = lope.apply_batch(grids, st, ins, nsteps=T, launch=launch)
        torch.cuda.synchronize()
        lope.sync_status()
        for g, u, o in zip(grids, ins, outs):
            ref = lope.apply(g, st, u, nsteps=T, launch=lope.Launch(DIRECT, 0, 0, 0, -1))
            assert torch.equal(ref, o), (g.shape, T)

    for k in depths:
        once(k, lope.Launch(STRIP, 0, 0, k, -1))
        once(2 * k + 1, lope.Launch(STRIP, 0, 0, k, -1))
    for _ in range(2):
        once(15, None)
        torch.cuda.empty_cache()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("shape", [(3, 64, 64), (9, 65, 68), (20, 120, 120), (50, 177, 236), (33, 64, 612)],
                         ids=lambda s: "x".join(map(str, s)))
def test_bricks_bitwise_equal_direct(lope, shape, dtype):
    """The 3D form: one to several blocks per axis, chunks shorter and longer
    than the pipeline, each axis periodic or Dirichlet with zero and non-zero
    values, sweep counts that end on depths 4, 2 and 1."""
    st = lope.Stencil.builtin("diff7", 0.1)
    u, _ = to_device(LI.uniform_field(1860, shape), dtype)
    for bcs in ([0, 0, 0], [1, 1, 1], [1, 0, 1], [0, 1, 0], [0, 0, 1]):
        for bv in (None, [(0.3, -0.2), (0.1, 0.5), (-0.4, 0.7)]):
            g = lope.Grid(shape, dtype, halo=1).set_boundaries(bcs, bv)
            for T, k in ((4, 4), (2, 2), (7, 4), (3, 2)):
                _check(lope, g, st, [u], T, k)


@pytest.mark.parametrize("shape", [(5, 64, 65), (20, 121, 127), (31, 70, 301)], ids=lambda s: "x".join(map(str, s)))
def test_bricks_rows_of_any_pitch_and_tables(lope, shape):
    rng = np.random.default_rng(1861)
    w = np.zeros((3, 3, 3))
    for i in ((0, 1, 1), (2, 1, 1), (1, 0, 1), (1, 2, 1), (1, 1, 0), (1, 1, 2)):
        w[i] = rng.uniform(0.02, 0.12)
    w[1, 1, 1] = 1.0 - w.sum()
    u, _ = to_device(LI.uniform_field(1862, shape), "f32")
    for st in (lope.Stencil.builtin("diff7", 0.1), lope.Stencil.linear(w)):
        for bcs in ([0, 0, 0], [1, 1, 1], [1, 0, 1], [0, 1, 0]):
            g = lope.Grid(shape, "f32", halo=1).set_boundaries(bcs, [0.5 if b else 0.0 for b in bcs])
            _check(lope, g, st, [u], 9, 4)


def test_bricks_write_only_their_output(lope):
    shape = (21, 70, 133)
    n = int(np.prod(shape))
    guard, sentinel = 4096, -7.0e30
    u = torch.rand(shape, device="cuda")
    keep = u.clone()
    st = lope.Stencil.builtin("diff7", 0.1)
    for bc in ([0, 0, 0], [1, 1, 1]):
        g = lope.Grid(shape, "f32", halo=1).set_boundaries(bc)
        bufs = [torch.full((n + 2 * guard,), sentinel, device="cuda") for _ in range(2)]
        out, work = (b[guard:guard + n].view(shape) for b in bufs)
        lope.apply(g, st, u, out=out, work=work, nsteps=10, launch=lope.Launch(STRIP, 0, 0, 4, -1))
        torch.cuda.synchronize()
        for b in bufs:
            assert bool((b[:guard] == sentinel).all()) and bool((b[guard + n:] == sentinel).all())
        assert torch.equal(u, keep)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("T,ckpt", [(23, 10), (13, 7), (6, 6), (9, 1)])
def test_brick_adjoint_equals_one_step_kernels(lope, orc, dtype, bc, T, ckpt):
    """diff7 on a grid large enough for the bricks: dL/du0 bitwise that of the
    same steps one at a time (the forward sweeps of a function equal to its own
    transpose), dL/dc the sum of <lambda, L u_t> to FP32 rounding of its terms."""
    shape, c = (65, 256, 256), 0.1
    u, _ = to_device(LI.uniform_field(1870, shape), dtype)
    gT, _ = to_device(LI.normal_field(1871, shape), dtype)
    st = lope.Stencil.builtin("diff7", c)
    g = lope.Grid(shape, dtype, halo=1).set_boundaries([bc] * 3)
    grad, gc = lope.vjp(g, st, u, gT, T, ckpt)
    torch.cuda.synchronize()
    lope.sync_status()
    ref = _run(lope, g, st, gT, T, lope.Launch(DIRECT, 0, 0, 0, -1))
    assert torch.equal(grad, ref)
    # the sum in FP64 from the stored states: L u_t = (u_{t+1} - u_t) / c up to
    # the rounding of the stored state, so evaluate L itself
    def lap(x):
        x = x.double()
        if bc:
            p = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
        else:
            p = torch.nn.functional.pad(x[None, None], (1, 1, 1, 1, 1, 1), mode="circular")[0, 0]
        s = p[2:, 1:-1, 1:-1] + p[:-2, 1:-1, 1:-1] + p[1:-1, 2:, 1:-1] + p[1:-1, :-2, 1:-1]
        return s + p[1:-1, 1:-1, 2:] + p[1:-1, 1:-1, :-2] - 6.0 * x
    lam, total, scale = gT, 0.0, 0.0
    states = [u]
    for _ in range(T - 1):
        states.append(_run(lope, g, st, states[-1], 1, lope.Launch(DIRECT, 0, 0, 0, -1)))
    for t in range(T - 1, -1, -1):
        l = lap(lam)
        total += float((l * states[t].double()).sum())
        scale += float((lam.double().abs() * states[t].double().abs()).sum())
        lam = _run(lope, g, st, lam, 1, lope.Launch(DIRECT, 0, 0, 0, -1))
    # each term: 7 roundings of sums of at most 12 |lambda| |u|, then a chain of
    # 4 FMAs and 2 adds in FP32 before FP64 takes over
    assert abs(float(gc) - total) <= 12 * 13 * 2.0 ** -24 * scale


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("T,ckpt", [(2, 2), (2, 5), (3, 3), (4, 2)])
def test_brick_adjoint_in_place(lope, dtype, T, ckpt):
    """lope_vjp with the gradient written over the upstream gradient: the values
    of separate buffers (two steps in all would be one pass that reads cells of
    one block while another writes them)."""
    shape = (65, 256, 256)
    u, _ = to_device(LI.uniform_field(1872, shape), dtype)
    gT, _ = to_device(LI.normal_field(1873, shape), dtype)
    st = lope.Stencil.builtin("diff7", 0.1)
    g = lope.Grid(shape, dtype, halo=1)
    want, gc = lope.vjp(g, st, u, gT, T, ckpt)
    ws = torch.empty(lope.workspace_size(g, st, T, ckpt), dtype=torch.uint8, device="cuda")
    got, gc2 = gT.clone(), torch.zeros(1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    lope.lope_vjp(g.handle, st.handle, u.data_ptr(), got.data_ptr(), T, ckpt, 0, got.data_ptr(),
                  gc2.data_ptr(), ws.data_ptr(), ws.numel(), 0)
    torch.cuda.synchronize()
    lope.sync_status()
    assert torch.equal(got, want)
    # dL/dc: the same terms, whichever steps share a pass, to the FP32 rounding of
    # each (independent errors: L^T lambda rounds 7 times on sums of 12 |lambda|)
    assert abs(float(gc2) - float(gc)) <= 100 * 2.0 ** -24 * float((T * gT.double().square().sum()).sqrt())


def _dlap(x, bcs):
    """L x in FP64 (Dirichlet 0 or periodic per axis), and the sum of the magnitudes
    of its terms."""
    p = x.double()
    for ax in range(3):
        if bcs[ax]:
            z = torch.zeros_like(p.narrow(ax, 0, 1))
            p = torch.cat([z, p, z], ax)
        else:
            p = torch.cat([p.narrow(ax, p.shape[ax] - 1, 1), p, p.narrow(ax, 0, 1)], ax)
    def star(q):
        return (q[2:, 1:-1, 1:-1] + q[:-2, 1:-1, 1:-1] + q[1:-1, 2:, 1:-1] + q[1:-1, :-2, 1:-1]
                + q[1:-1, 1:-1, 2:] + q[1:-1, 1:-1, :-2])
    return star(p) - 6.0 * x.double(), star(p.abs()) + 6.0 * x.double().abs()


def _dc(lope, g, st, u, lam, T, bcs):
    """dL/dc in FP64 from the stored states of single steps, the root of the sum of
    the squared magnitudes of its terms, and dL/du0."""
    one = lope.Launch(DIRECT, 0, 0, 0, -1)
    states, total, square = [u], 0.0, 0.0
    for _ in range(T - 1):
        states.append(_run(lope, g, st, states[-1], 1, one))
    for t in range(T - 1, -1, -1):
        l, size = _dlap(lam, bcs)
        total += float((l * states[t].double()).sum())
        square += float((size * states[t].double()).square().sum())
        lam = _run(lope, g, st, lam, 1, one)
    return total, square ** 0.5, lam


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("shape,bcs", [((37, 380, 300), [1, 0, 1]), ((37, 380, 300), [0, 1, 0]),
                                       ((130, 189, 204), [0, 0, 1]), ((130, 189, 204), [1, 1, 0]),
                                       ((126, 200, 300), [1, 1, 1])], ids=str)
@pytest.mark.parametrize("T,ckpt", [(13, 7), (4, 4)])
def test_brick_adjoint_counts_every_cell_once(lope, dtype, shape, bcs, T, ckpt):
    """dL/dc on extents that are no multiple of a block's, sides of both kinds:
    each term rounds at most 12 times (7 in L^T lambda, a chain of 4 FMAs, one
    sum), independently, so four deviations of the sum are 4 * 12 / sqrt(3) *
    2^-24 of the root sum square; a single missing cell is a hundred times that."""
    u, _ = to_device(LI.uniform_field(1890, shape), dtype)
    gT, _ = to_device(LI.normal_field(1891, shape), dtype)
    st = lope.Stencil.builtin("diff7", 0.1)
    g = lope.Grid(shape, dtype, halo=1).set_boundaries(bcs)
    grad, gc = lope.vjp(g, st, u, gT, T, ckpt)
    torch.cuda.synchronize()
    lope.sync_status()
    total, size, lam = _dc(lope, g, st, u, gT, T, bcs)
    assert torch.equal(grad, lam)
    assert abs(float(gc) - total) <= 28 * 2.0 ** -24 * size


def test_brick_adjoint_sum_has_the_range_of_fp64(lope):
    """Terms whose sum passes FP32's largest value while those of a row do not: the
    second difference of lambda along x is +1 or -1, and u has its sign."""
    shape, bcs, T = (65, 256, 256), [0, 0, 0], 2
    s = np.where((np.arange(256) < 64) | (np.arange(256) >= 192), 1.0, -1.0)
    slope = np.cumsum(s)
    lam = np.concatenate([[0.0], np.cumsum(slope - slope.mean())[:-1]])  # exact: halves below 2^13
    assert np.array_equal(np.roll(lam, -1) + np.roll(lam, 1) - 2 * lam, s)
    gT = torch.from_numpy(lam * 2.0 ** 57).float().cuda().expand(shape).contiguous()
    u = torch.from_numpy(s * 2.0 ** 66).float().cuda().expand(shape).contiguous()
    st = lope.Stencil.builtin("diff7", 0.1)
    g = lope.Grid(shape, "f32", halo=1).set_boundaries(bcs)
    _, pairs = lope.vjp(g, st, u, gT, T, 2)   # one pass of two steps
    _, single = lope.vjp(g, st, u, gT, T, 1)  # one step per pass: the same L^T lambda
    torch.cuda.synchronize()
    lope.sync_status()
    # Only the sums differ: either rounds a term at most 5 times before FP64 takes it.
    one = lope.Launch(DIRECT, 0, 0, 0, -1)
    u1, lam1 = _run(lope, g, st, u, 1, one), _run(lope, g, st, gT, 1, one)
    terms = sum(float((_dlap(l, bcs)[0] * v.double()).abs().sum()) for l, v in ((gT, u1), (lam1, u)))
    assert float(single) > 1e40
    assert abs(float(pairs) - float(single)) <= 10 * 2.0 ** -24 * 1.01 * terms


@pytest.mark.parametrize("shape,name,prm,T", [((100, 200), "jacobi5", [0.2], 20), ((64, 256, 256), "diff7", [0.1], 16),
                                              ((130, 100, 130), "diff7", [0.1], 16)], ids=str)
def test_autotuner_keeps_a_faster_plan_of_the_planner(lope, shape, name, prm, T):
    """The strips and bricks run these calls in about half the time of the tiles:
    after tuning they still do, with the same result."""
    st = lope.Stencil.builtin(name, *prm)
    g = lope.Grid(shape, "f32", halo=1).set_boundaries([1] * len(shape))
    u = torch.rand(shape, device="cuda")
    o, w = torch.empty_like(u), torch.empty_like(u)
    want = _run(lope, g, st, u, T, None)
    best, ms = lope.autotune(g, st, u, o, w, T)
    assert ms > 0 and best.path in (1, 2, 3, 4, STRIP)
    assert lope.plan(g, st, u, o, w, nsteps=T)[0].path == STRIP
    assert torch.equal(_run(lope, g, st, u, T, None), want)


@pytest.mark.parametrize("name,prm,halo", [("jacobi5", [0.2], 1), ("star9r2", [0.1], 2)])
def test_batch_autotuner_keeps_a_faster_plan(lope, name, prm, halo):
    """Likewise for a batch below 2^20 points (strips: one kernel per pass and one
    for the descriptors; trapezoid tiles: two kernels).  Radius 2 has no other form."""
    st = lope.Stencil.builtin(name, *prm)
    shapes = [(64 + 15 * i, 300 - 13 * i) for i in range(16)]
    grids = [lope.Grid(s, "f32", halo=halo) for s in shapes]
    ins = [torch.rand(s, device="cuda") for s in shapes]
    outs, works = [torch.empty_like(x) for x in ins], [torch.empty_like(x) for x in ins]

    def kernels():
        n = lope.launch_count()
        lope.apply_batch(grids, st, ins, outs, works, nsteps=20)
        return lope.launch_count() - n

    before = kernels()
    assert before > 2
    best, ms = lope.autotune_batch(grids, st, ins, outs, works, 20)
    assert ms > 0
    assert kernels() == before
    torch.cuda.synchronize()
    lope.sync_status()


@pytest.mark.parametrize("kinds,passes", [([0, 0], 3), ([0, 1], 5), ([1, 1], 5)])
def test_depth_of_radius_two_batches(lope, kinds, passes):
    """Nine sweeps of star9r2: 4 + 4 + 1 on periodic grids, 2 + 2 + 2 + 2 + 1 where a grid
    has Dirichlet sides, after one kernel for the descriptors; each grid as alone."""
    st = lope.Stencil.builtin("star9r2", 0.1)
    shapes = [(70, 133), (300, 224)]
    grids = [lope.Grid(s, "f32", halo=2).set_boundaries([k, k]) for s, k in zip(shapes, kinds)]
    ins = [torch.rand(s, device="cuda") for s in shapes]
    n = lope.launch_count()
    outs = lope.apply_batch(grids, st, ins, nsteps=9)
    assert lope.launch_count() - n == passes + 1
    for g, u, o in zip(grids, ins, outs):
        assert torch.equal(_run(lope, g, st, u, 9, lope.Launch(DIRECT, 0, 0, 0, -1)), o)


@pytest.mark.parametrize("dtype,shape,bcs,pairs", [
    ("f32", (65, 256, 256), [1, 1, 1], False), ("f32", (65, 256, 256), [1, 0, 1], True),
    ("f32", (65, 256, 256), [0, 0, 0], True), ("f32", (128, 200, 300), [1, 1, 1], True),
    ("bf16", (128, 256, 256), [1, 1, 1], False), ("bf16", (128, 256, 256), [1, 0, 1], True),
    ("bf16", (65, 256, 256), [1, 0, 1], False), ("bf16", (40, 600, 600), [1, 1, 1], True)], ids=str)
def test_route_of_the_adjoint(lope, dtype, shape, bcs, pairs):
    """Four steps back from one checkpoint: in pairs (zeroing, states 2 + 1, two passes,
    the final sum) or one at a time (zeroing, 3 states, 4 steps, the final sum),
    whichever is faster there."""
    st = lope.Stencil.builtin("diff7", 0.1)
    g = lope.Grid(shape, dtype, halo=1).set_boundaries(bcs)
    u, _ = to_device(LI.uniform_field(1900, shape), dtype)
    gT, _ = to_device(LI.normal_field(1901, shape), dtype)
    _, ws = lope.forward_ckpt(g, st, u, 4, 4)
    n = lope.launch_count()
    grad, _ = lope.vjp(g, st, u, gT, 4, 4, reuse=True, workspace=ws)
    assert lope.launch_count() - n == (6 if pairs else 9)
    assert torch.equal(grad, _run(lope, g, st, gT, 4, lope.Launch(DIRECT, 0, 0, 0, -1)))
