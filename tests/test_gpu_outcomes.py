"""What the calls tell their callers, and results at the ends of FP32's range (GB300)."""

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
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _phi(shape, seed):
    rng = np.random.default_rng(seed)
    return np.where(rng.uniform(size=shape) < 0.35, -1, 1).astype(np.float32)


@pytest.mark.parametrize("prec", ["fp32", "mixed_bf16"])
def test_preconditioner_reports_a_wait_that_ran_out(ext, prec):
    """A wait bound of one cycle: the kernels drain and return, and the call itself says so."""
    c = ext.ext_create(ext.options(prec, wait_cycles=1))
    try:
        r2, r3 = torch.ones((150, 200), device="cuda"), torch.ones((128,) * 3, device="cuda")
        for call, prob, r in ((ext.ext_apply_preconditioner, ext.problem(200, 150), r2),
                              (ext.ext_apply_preconditioner3d, ext.problem3(128, 128, 128), r3)):
            with pytest.raises(ext.ExtError) as e:
                call(c, prob, torch.ones_like(r), r, torch.empty_like(r))
            assert e.value.code == ext.EXT_ETIMEOUT
    finally:
        ext.ext_destroy(c)


@pytest.mark.parametrize("prec,kw", [("fp32", {}), ("mixed_bf16", {}), ("mixed_fp16", dict(low_modes=0)),
                                     ("mixed_bf16", dict(low_modes=1))])
@pytest.mark.parametrize("shape", [(70, 60), (250, 300), (128, 128, 128)])
def test_preconditioner_of_a_small_residual(ext, prec, kw, shape):
    """Residuals far below one against the oracle's box solve, within the bound of the other preconditioner
    tests at magnitude one, 5e-6 of the largest entry.  (What FP32's range takes is below that down to
    1e-31: an element of r or T1..T3 is off by 2^-143 at most, one of z by 4 sqrt(N) 2^-143.)"""
    phi = _phi(shape, 5)
    r0 = np.where(phi < 0, 0, np.random.default_rng(6).standard_normal(shape))
    two = len(shape) == 2
    bcs = ("symmetric", "dirichlet") if two else ("symmetric", "dirichlet", "periodic")
    prob = ext.problem(*shape[::-1], *bcs) if two else ext.problem3(*shape[::-1], *bcs)
    call = ext.ext_apply_preconditioner if two else ext.ext_apply_preconditioner3d
    c = ext.ext_create(ext.options(prec, **kw))
    try:
        for size in (1.0, 1e-25, 1e-28, 1e-31):
            r = (r0 * size).astype(np.float32)
            z = torch.empty(shape, device="cuda")
            scale = call(c, prob, dev(phi), dev(r), z)
            r = r.astype(np.float64)
            ref = ob.poisson_squared_pinv(r, *bcs) if two else o3.poisson_squared_pinv3(r, bcs)
            ref[phi < 0] = 0
            np.testing.assert_allclose(z.cpu().numpy().astype(np.float64) / scale, ref, rtol=0,
                                       atol=5e-6 * np.abs(ref).max(), err_msg=f"magnitude {size}")
    finally:
        ext.ext_destroy(c)


@pytest.mark.parametrize("size", ["1", "1e-25", "1e20", "1e-40", "spread"])
@pytest.mark.parametrize("nx,ny", [(5, 4), (65, 17), (700, 430)])
def test_sum_of_the_operator_without_a_context(ext, nx, ny, size):
    """p.q against the exact sum of the products p q of the q returned.  Tolerance: a tile's and the call's
    sums are FP64, at most 4 + 5 + 8 + 30 additions deep (512 x 512 nodes; a thread's, a warp's, a block's,
    the tiles'), each 2^-53 of the sum of magnitudes: 47 2^-53."""
    from fractions import Fraction
    rng = np.random.default_rng(nx)
    p = rng.standard_normal((ny, nx))
    p = p * (10.0 ** rng.uniform(-30, 15, (ny, nx)) if size == "spread" else float(size))
    phi = _phi((ny, nx), 2)
    p[phi < 0] = 0
    p = p.astype(np.float32)
    q = torch.empty((ny, nx), device="cuda")
    rc, got = ext.ext_apply_biharmonic_noalloc(ext.problem(nx, ny, "symmetric", "periodic"), dev(phi), dev(p), q)
    assert rc == ext.EXT_OK
    terms = [Fraction(float(a)) * Fraction(float(b)) for a, b in zip(p.ravel(), q.cpu().numpy().ravel()) if a and b]
    want, size_of = sum(terms), sum(abs(t) for t in terms)
    assert size_of > 0 and abs(Fraction(got) - want) <= 47 * size_of / 2 ** 53


@pytest.mark.parametrize("tile_y", [16, 32])
def test_direction_sums_are_fp64_across_warps(ext, tile_y):
    """p.q of the stencil, one 64 x 16 block: a single node of p per warp, three columns apart, so that
    each warp's sum is one product 20 p^2, exact in a pair of FP32 numbers; the eight together span 53 bits,
    exact in FP64 and not in such a pair."""
    nx, ny = 64, 16
    p = np.zeros((ny, nx), np.float32)
    vals = [(2 ** 19 - 1) * 2 ** 6] + [2 ** 19 - 1 - 2 * k for k in range(1, 6)]
    for w, v in enumerate(vals):
        p[2 + w, 4 + 6 * w] = v  # rows 2..7: the warps that hold them, away from the edges
    q = torch.empty((ny, nx), device="cuda")
    c = ext.ext_create(ext.options("fp32", autotune=0, tile_y=tile_y))
    try:
        got = ext.ext_apply_biharmonic(c, ext.problem(nx, ny), dev(np.ones_like(p)), dev(p), q)
    finally:
        ext.ext_destroy(c)
    want = 20 * sum(v * v for v in vals)
    assert want.bit_length() - 2 <= 53 and int(got) == want, (got, want)


@pytest.mark.parametrize("prec,kw", [("fp32", {}), ("mixed_bf16", {}), ("mixed_bf16", dict(low_modes=1))])
@pytest.mark.parametrize("nx,ny", [(70, 61), (130, 140), (389, 251), (300, 257)])
def test_a_residual_of_nans_leaves_nothing_behind(ext, prec, kw, nx, ny):
    """The transform stages' operands share memory: after a residual of NaNs the same context gives a finite
    one the z that a fresh context gives, bit for bit."""
    phi = _phi((ny, nx), 3)
    r = np.where(phi < 0, 0, np.random.default_rng(4).standard_normal((ny, nx))).astype(np.float32)
    prob = ext.problem(nx, ny, "symmetric", "dirichlet")
    zs = []
    for before in ([], [np.full_like(r, np.nan), np.full_like(r, np.inf)]):
        c = ext.ext_create(ext.options(prec, **kw))
        try:
            z = torch.empty((ny, nx), device="cuda")
            for bad in before:
                ext.ext_apply_preconditioner(c, prob, dev(phi), dev(bad), z)
                assert not torch.isfinite(z).all()
            ext.ext_apply_preconditioner(c, prob, dev(phi), dev(r), z)
        finally:
            ext.ext_destroy(c)
        zs.append(z)
    assert torch.isfinite(zs[0]).all() and torch.equal(*zs)
