"""The rules that choose a kernel by size (GB300): each call on one side of a rule against the same
grid on the other side, or against the oracle, at the edges of the rules and of the tiles.

* A grid's solve does not depend on what else is in the call: alone (update that slices the residual,
  scalars formed by their consumers) and among other grids (a grid above 2^17 nodes in the call: plain
  update and separate slicing; more than eight grids: separate scalar kernels; more tiles than SMs: work
  lists with empty places) the iterates are the same bit for bit.  The comparison is exact: both sides
  evaluate the same sums in the same order.  Sides: odd (a middle row and column in the even classes), of
  whole 16-byte vectors or not, folded on both axes, one or none; both sides of 2^17 nodes and of the
  line between six and four slices (768^2 nodes).
* The 3-D transform products at the edges of their 32 x 32 tiles against the oracle's box solve.
  Tolerance: three products of at most n <= 80 FP32 terms a row and back, 6 n 2^-24 = 3e-5 worst
  case relative to the largest entry; a random sum's error grows as its square root, 6 sqrt(n) 2^-24 =
  3.2e-6: 5e-6, the bound of the other 3-D preconditioner tests.
* The operator without a context against the context's at the edges of its 64 x 16 tiles: q bit for bit.
"""

import numpy as np
import pytest

from oracle import biharmonic as ob
from oracle import biharmonic3d as o3

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ext():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1704_08897_gb300 import build_ext, ext as e
    build_ext.build()
    e.load()
    return e


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _problem(ext, nx, ny, seed):
    rng = np.random.default_rng(seed)
    X, Y = np.meshgrid(np.linspace(-1, 1, nx), np.linspace(-1, 1, ny))
    phi = np.hypot(X - 0.1, Y + 0.05) - 0.5 - 0.06 * np.cos(5 * np.arctan2(Y, X))
    f = np.cos(3 * X + rng.uniform(0, 3)) * np.sin(2 * Y) + 0.3 * X * Y
    bc = list(rng.choice(ob.BCS, 2))
    return (ext.problem(nx, ny, *bc, ["out", "in"][seed % 2]), dev(phi.astype(np.float32)),
            dev(f.astype(np.float32)))


@pytest.mark.parametrize("prec", ["mixed_bf16", "mixed_fp16", "fp32"])
@pytest.mark.parametrize("sides", [
    # small grids with one above 2^17 nodes
    [(64, 64), (65, 33), (389, 251), (300, 131), (255, 200), (400, 340)],
    # 2^17 nodes and just above
    [(512, 256), (512, 257)],
    # more than eight grids, all small
    [(4, 4), (24, 40), (33, 64), (130, 60), (97, 97), (128, 129), (200, 256), (254, 66), (18, 300), (386, 260)],
    # more tiles than SMs
    [(500, 500)] * 3 + [(260, 300)] * 5 + [(128, 128)],
], ids=["one-large", "edge-2^17", "ten-small", "many-tiles"])
def test_a_grid_solves_the_same_in_any_company(ext, prec, sides):
    # bf16: six slices up to 768^2 nodes (automatic); fp16: four everywhere
    c = ext.ext_create(ext.options(prec, rtol=1e-5, maxit=60, low_modes=0 if prec == "mixed_fp16" else 2))
    try:
        cases = [_problem(ext, nx, ny, i) for i, (nx, ny) in enumerate(sides)]
        single = []
        for prob, phi, f in cases:
            out = torch.empty_like(f)
            single.append((ext.ext_solve(c, prob, phi, f, out, check=False), out))
        outs = [torch.empty_like(f) for _, _, f in cases]
        _, res = ext.ext_solve_batch(c, [k[0] for k in cases], [k[1] for k in cases], [k[2] for k in cases],
                                     outs, check=False)
        for (r1, o1), r2, o2, s in zip(single, res, outs, sides):
            assert r1["iters"] == r2["iters"] > 0 and r1["status"] == r2["status"], (s, r1, r2)
            assert torch.isfinite(o1).all() and torch.equal(o1, o2), s
    finally:
        ext.ext_destroy(c)


def test_slices_by_grid_size_do_not_depend_on_company(ext):
    """768 x 768 nodes (six slices), one row more (four), and a small grid, alone and together."""
    c = ext.ext_create(ext.options("mixed_bf16", rtol=1e-5, maxit=20))
    try:
        cases = [_problem(ext, nx, ny, i) for i, (nx, ny) in enumerate([(768, 768), (768, 769), (100, 100)])]
        single = []
        for prob, phi, f in cases:
            out = torch.empty_like(f)
            ext.ext_solve(c, prob, phi, f, out, check=False)
            single.append(out)
        outs = [torch.empty_like(f) for _, _, f in cases]
        ext.ext_solve_batch(c, [k[0] for k in cases], [k[1] for k in cases], [k[2] for k in cases], outs, check=False)
        for o1, o2 in zip(single, outs):
            assert torch.isfinite(o1).all() and torch.equal(o1, o2)
    finally:
        ext.ext_destroy(c)


@pytest.mark.parametrize("shape", [(31, 33, 65), (32, 64, 32), (80, 31, 4)])
@pytest.mark.parametrize("bcs", [("symmetric", "periodic", "dirichlet"), ("dirichlet", "symmetric", "periodic")])
def test_3d_products_at_the_edges_of_their_tiles(ext, bcs, shape):
    nz, ny, nx = shape
    rng = np.random.default_rng(3)
    phi = np.where(rng.uniform(size=shape) < 0.35, rng.uniform(-1, 1, shape), 1.0).astype(np.float32)
    unk = ~ob.known_mask(phi.astype(np.float64), "out")
    r = np.where(unk, rng.standard_normal(shape), 0).astype(np.float32)
    ref = np.where(unk, o3.poisson_squared_pinv3(r.astype(np.float64), bcs), 0.0)
    c = ext.ext_create(ext.options("fp32", rtol=1e-8))
    try:
        z = torch.empty(shape, device="cuda")
        scale = ext.ext_apply_preconditioner3d(c, ext.problem3(nx, ny, nz, *bcs, "out"), dev(phi), dev(r), z)
    finally:
        ext.ext_destroy(c)
    np.testing.assert_allclose(z.cpu().numpy().astype(np.float64) / scale, ref, rtol=0, atol=5e-6 * np.abs(ref).max())


@pytest.mark.parametrize("nx,ny", [(4, 4), (63, 15), (64, 16), (65, 17), (1024, 1024)])
@pytest.mark.parametrize("h", [(1.0, 1.0), (0.02, 0.03)])
def test_operator_without_a_context_at_tile_edges(ext, nx, ny, h):
    rng = np.random.default_rng(nx + ny)
    phi = rng.uniform(-1, 1, (ny, nx)).astype(np.float32)
    p = np.where(phi < 0, 0, rng.standard_normal((ny, nx))).astype(np.float32)
    prob = ext.problem(nx, ny, "symmetric", "dirichlet", "out", *h)
    c = ext.ext_create(ext.options("fp32"))
    try:
        want = torch.empty((ny, nx), device="cuda")
        ext.ext_apply_biharmonic(c, prob, dev(phi), dev(p), want)
    finally:
        ext.ext_destroy(c)
    q = torch.full((ny, nx), float("nan"), device="cuda")
    rc, _ = ext.ext_apply_biharmonic_noalloc(prob, dev(phi), dev(p), q)
    assert rc == ext.EXT_OK and torch.equal(q, want)
