"""The plans of calls of 12 and more sweeps (plan queries: fake addresses, no GPU).

The register strips run nearly all 2D calls at their deepest; the shapes here are
those that measured faster at another depth, or on the plan of shorter calls.
"""
import numpy as np
import pytest

TMA, TRAP, STRIP = 1, 2, 5
P, D = 0, 1
PRM = {"jacobi5": ([0.2], 1, 1), "star9r2": ([0.1], 2, 1), "diff7": ([0.1], 1, 1),
       "swe_cgrid": ([0.02, 1.0, 1.0], 1, 3), "swe_flux": ([0.02, 1.0, 0.5, 1.0], 1, 3)}
CROSS2 = """
for (int f = 0; f < NF; ++f)
  out[f] = fma_(P[0], sub(add(U(f, -2, 0), U(f, 0, 2)), add(U(f, 2, 0), U(f, 0, -2))), U(f, 0, 0));
"""


def _plan(L, shape, dtype, fn, bc, steps=12, scheme="euler", tile=False):
    """(path, depth) of a call with aligned pointers; tile: (path, tile, depth)."""
    if fn == "box2":
        w = np.arange(1.0, 26.0).reshape(5, 5) / 325.0
        st, halo, nf = L.Stencil.linear(w), 2, 1
    elif fn.startswith("user"):
        nf, halo = int(fn[4]), 2
        st = L.Stencil.source(CROSS2, ndim=2, radius=2, nfields=nf, params=[0.05])
    else:
        prm, halo, nf = PRM[fn]
        st = L.Stencil.builtin(fn, *prm)
    if scheme != "euler":
        st.set_scheme(scheme)
    g = L.Grid(shape, dtype, halo=halo, nfields=nf).set_boundaries(bc)
    field = (int(np.prod(shape)) * {"f32": 4, "f64": 8, "bf16": 2}[dtype] + 255) // 256 * 256
    base = 1 << 44
    at = lambda k: [base + (k * nf + f) * 2 * field for f in range(nf)]  # noqa: E731
    plan, _ = L.lope_plan(g.handle, st.handle, at(0), at(1), at(2), steps, None)
    if tile:
        return plan.path, plan.tile_x, plan.tile_y, plan.tsteps
    return plan.path, plan.tsteps


@pytest.mark.parametrize("fn,dtype,shape,bc,want", [
    ("jacobi5", "f32", (1000, 1000), [D, D], (STRIP, 8)),
    ("swe_cgrid", "f32", (1000, 1000), [D, D], (STRIP, 6)),
    # radius-2 box tables
    ("box2", "f32", (300, 300), [P, P], (STRIP, 2)),
    ("box2", "f32", (300, 300), [D, D], (TRAP, 4)),
    ("box2", "f32", (60, 8192), [D, D], (TRAP, 4)),
    ("box2", "f32", (1000, 1000), [D, D], (STRIP, 2)),
    ("box2", "f32", (600, 603), [D, D], (TRAP, 4)),
    ("box2", "f32", (2000, 2003), [D, D], (STRIP, 2)),
    ("box2", "f32", (2000, 2000), [P, P], (TMA, 1)),
    ("box2", "f32", (4096, 4096), [D, D], (TMA, 2)),
    ("box2", "bf16", (4096, 4096), [D, D], (TMA, 1)),
    ("box2", "bf16", (2000, 2000), [D, D], (STRIP, 2)),
    # states that the tiles read from L2, with masks
    ("swe_flux", "f32", (1000, 1000), [D, D], (TMA, 1)),
    ("swe_flux", "f32", (1000, 1000), [D, P], (STRIP, 4)),
    ("swe_flux", "f32", (1000, 1003), [D, D], (STRIP, 4)),
    ("swe_flux", "f32", (3000, 3000), [D, D], (STRIP, 4)),
    ("swe_flux", "f32", (600, 603), [D, D], (STRIP, 2)),
    ("swe_flux", "bf16", (1200, 1200), [D, D], (TMA, 1)),
    ("swe_flux", "bf16", (1000, 1000), [D, D], (STRIP, 4)),
    ("star9r2", "f32", (2000, 2000), [D, D], (TMA, 1)),
    ("star9r2", "f32", (2000, 2000), [P, P], (STRIP, 4)),
    ("star9r2", "f32", (4096, 4096), [D, D], (STRIP, 4)),
    # run-time compiled functions of radius 2
    ("user3", "f32", (1000, 1000), [P, P], (TMA, 1)),
    ("user3", "f32", (300, 300), [D, P], (TRAP, 4)),
    ("user3", "f32", (4096, 4096), [P, P], (STRIP, 2)),
    ("user2", "f32", (4096, 4096), [P, P], (STRIP, 4)),
    ("user2", "f32", (4096, 4096), [D, D], (STRIP, 2)),
], ids=str)
def test_depth_of_long_calls(lope, fn, dtype, shape, bc, want):
    assert _plan(lope, shape, dtype, fn, bc) == want


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("shape,bc,want", [
    ((16, 512, 512), [D, D, D], (TMA, 2)),
    ((24, 512, 512), [P, D, D], (TMA, 2)),
    ((40, 512, 512), [D, D, D], (STRIP, 4)),
    ((16, 512, 512), [P, P, P], (STRIP, 4)),
    ((16, 304, 1000), [D, D, D], (STRIP, 4)),
    ((16, 4096, 64), [D, D, D], (STRIP, 4)),
    ((64, 64, 64), [D, D, D], (TMA, 1)),
], ids=str)
def test_bricks_on_thin_grids(lope, dtype, shape, bc, want):
    """Thin grids whose blocks leave half of the SMs idle keep two sweeps per launch
    where those run (x and y sides Dirichlet)."""
    assert _plan(lope, shape, dtype, "diff7", bc) == want


@pytest.mark.parametrize("fn,shape,want", [
    ("jacobi5", (256, 256), (64, 8, 4)), ("jacobi5", (100, 300), (32, 8, 4)),
    ("jacobi5", (426, 640), (64, 16, 4)), ("jacobi5", (511, 513), (64, 16, 4)),
    ("jacobi5", (512, 512), (32, 8, 1)), ("star9r2", (700, 900), (32, 8, 1)),
], ids=str)
def test_tile_of_double_grids(lope, fn, shape, want):
    """Another tile than 64 x 16 at depth 4 only where the estimate is clearly better."""
    assert _plan(lope, shape, "f64", fn, [D, P], tile=True) == (TRAP,) + want


@pytest.mark.parametrize("fn,dtype,shape,bc,scheme,path", [
    ("box2", "bf16", (1000, 1000), [D, D], "rk2", TMA),
    ("box2", "bf16", (1000, 1000), [P, P], "rk2", STRIP),
    ("box2", "bf16", (1000, 1000), [P, P], "rk3", TMA),
    ("box2", "bf16", (144, 600), [D, P], "rk3", TMA),
    ("box2", "bf16", (144, 600), [D, P], "rk2", STRIP),
    ("box2", "f32", (1000, 1000), [D, D], "rk3", STRIP),
    ("swe_flux", "f32", (848, 848), [D, D], "rk3", TMA),
    ("swe_flux", "f32", (848, 848), [P, P], "rk3", STRIP),
    ("swe_flux", "f32", (2000, 2000), [D, D], "rk3", STRIP),
], ids=str)
def test_path_of_long_multi_stage_calls(lope, fn, dtype, shape, bc, scheme, path):
    assert _plan(lope, shape, dtype, fn, bc, scheme=scheme)[0] == path
