"""The library's host code on the CPU, over a CUDA runtime without a device (fake_cuda/cudart.cu): what
the host does around the kernels, which no result on a GPU shows reliably."""

import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes as C, itertools, sys
import numpy as np
sys.path.insert(0, {root!r})
from paper_1704_08897_gb300 import ext
fake = C.CDLL({fake!r})
fake.fake_fail_malloc.argtypes = [C.c_long]
fake.fake_mallocs.restype = C.c_long
fake.fake_live_bytes.restype = C.c_size_t
rt = C.CDLL({fake!r})
class Dev:  # an array in "device" memory
    def __init__(self, n, itemsize=4):
        p = C.c_void_p()
        rt.cudaMalloc(C.byref(p), C.c_size_t(n * itemsize))
        C.memset(p, 0, n * itemsize)
        self.p = p.value
    def is_contiguous(self): return True
    def data_ptr(self): return self.p
def faults():
    b = C.create_string_buffer(1 << 16)
    fake.fake_faults(b, len(b))
    return b.value.decode()
"""


@pytest.fixture(scope="session")
def fake_cuda(tmp_path_factory):
    """Runs a script with the fake runtime in front; returns what it printed."""
    from paper_1704_08897_gb300 import build_ext, ext
    build_ext.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfakecudart.so")
    subprocess.run([build_ext._nvcc(), "-std=c++17", "-O1", *build_ext.ARCH, "--cudart", "none", "-shared",
                    "-Xcompiler", "-fPIC", "-diag-suppress", "177", os.path.join(HERE, "fake_cuda", "model.cu"),
                    os.path.join(HERE, "fake_cuda", "cudart.cpp"),
                    "-o", so], check=True, capture_output=True)

    def run(script):
        env = dict(os.environ, LD_PRELOAD=so)
        env.pop("EXT_TUNE_CACHE", None)
        p = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT, fake=so) + script], env=env,
                           capture_output=True, text=True, timeout=300)
        assert p.returncode == 0, p.stdout + p.stderr
        return p.stdout
    return run


# Every way into the library that sets something up for kernels on a stream of its own.
CALLS = """
def calls():
    phi, f, out = Dev(96 * 80), Dev(96 * 80), Dev(96 * 80)
    prob = ext.problem(96, 80, "symmetric", "periodic")
    for prec in ("fp32", "mixed_bf16"):
        for kw in (dict(), dict(autotune=0, tile_y=16), dict(low_modes=1)):
            c = ext.ext_create(ext.options(prec, **kw))
            yield "solve", lambda: ext.ext_solve(c, prob, phi, f, out, check=False)
            yield "batch", lambda: ext.ext_solve_batch(c, [prob] * 2, [phi] * 2, [f] * 2, [out] * 2, check=False)
            yield "served", lambda: (ext.ext_submit(c, prob, phi, f, out), ext.ext_drain(c))
            ext.ext_destroy(c)
            c = ext.ext_create(ext.options(prec, **kw))
            yield "operator", lambda: ext.ext_apply_biharmonic(c, prob, phi, f, out)
            ext.ext_destroy(c)
            c = ext.ext_create(ext.options(prec, **kw))
            yield "preconditioner", lambda: ext.ext_apply_preconditioner(c, prob, phi, f, out)
            ext.ext_destroy(c)
        for n in (12, 128):
            v = [Dev(n * n * 128) for _ in range(3)]
            p3 = ext.problem3(n, n, 128)
            for call in (ext.ext_apply_biharmonic3d, ext.ext_apply_preconditioner3d, ext.ext_solve3d):
                c = ext.ext_create(ext.options(prec))
                yield call.__name__, lambda: call(c, p3, *v)
                ext.ext_destroy(c)
"""


def test_set_up_is_complete_before_kernels_on_other_streams(fake_cuda):
    """Copies and memsets of the legacy stream may be in flight when their calls return, and the kernels'
    streams do not wait for that stream: each set-up has to wait before the first operation of another
    stream follows."""
    out = fake_cuda(CALLS + """
fake.fake_model(5, 3, 0)
for name, call in calls():
    call()
print(faults())
""")
    assert out.strip() == ""


@pytest.mark.parametrize("kw", ['dict(prec="mixed_bf16", low_modes=1, autotune=0)',
                                'dict(prec="mixed_bf16")', 'dict(prec="fp32", autotune=0, tile_y=16)'])
def test_a_failed_allocation_leaves_nothing_half_made(fake_cuda, kw):
    """Each allocation of a first call fails in turn: the call reports it, and the same call on the same
    context then works on complete plans and work lists (tensor maps, copies and lists inside live
    allocations)."""
    out = fake_cuda("""
phi, f, out = [Dev(160 * 256) for _ in range(3)]
v = [Dev(12 * 12 * 128) for _ in range(3)]
CALLS = [lambda c: ext.ext_solve(c, prob, phi, f, out, check=False)["rc"],
         lambda c: ext.load().ext_apply_preconditioner(c, C.byref(prob), phi.p, f.p, out.p, None),
         lambda c: ext.ext_solve3d(c, ext.problem3(12, 12, 128), *v, check=False)["rc"]]
told, kw = 0, """ + kw + """
for i, call in enumerate(CALLS):
    n = 0
    while True:
        fake.fake_fail_malloc(-1)
        c = ext.ext_create(ext.options(**kw))
        fake.fake_model(5, 2, 0)
        prob = ext.problem(160, 96 + n, "symmetric", "dirichlet")  # another height each time: none is tuned yet
        before = fake.fake_mallocs()
        fake.fake_fail_malloc(n)
        rc = call(c)
        failed = fake.fake_mallocs() - before > n
        fake.fake_fail_malloc(-1)
        fake.fake_model(5, 2, 0)
        if failed and rc not in (ext.EXT_ENOMEM, ext.EXT_ECUDA):
            print(kw, i, n, "failed allocation gave", rc)
        again = call(c)
        if len(faults()) != told:
            print(kw, i, n, rc, faults()[told:])
            told = len(faults())
        if again != ext.EXT_OK:
            print(kw, i, n, "the next call gave", again)
        ext.ext_destroy(c)
        if not failed:
            break
        n += 1
    assert n > 3, n
""")
    assert out.strip() == ""


def test_a_wait_that_runs_out_is_told_by_the_call_it_ran_out_in(fake_cuda):
    """Both preconditioner calls return EXT_ETIMEOUT when a transform product raises the flag, and the next
    call on the context starts with the flag down; a 3-D solve leaves after the block that raised it, not
    after all of its blocks."""
    out = fake_cuda("""
T = ext.EXT_ETIMEOUT
phi, f, z = [Dev(128 ** 3) for _ in range(3)]
prob, prob3 = ext.problem(200, 150), ext.problem3(128, 128, 128)
for prec in ("fp32", "mixed_bf16"):
    c = ext.ext_create(ext.options(prec, maxit=400))
    for name, call, p in (("2-D", ext.load().ext_apply_preconditioner, prob),
                          ("3-D", ext.load().ext_apply_preconditioner3d, prob3)):
        for err_after, want in ((1, T), (0, 0)):
            fake.fake_model(1, 0, err_after)
            rc = call(c, C.byref(p), phi.p, f.p, z.p, None)
            if rc != want: print(prec, name, err_after, rc)
    for err_after, ok_after, want in ((30, 0, T), (0, 5, 0)):
        fake.fake_model(1, ok_after, err_after)
        r = ext.ext_solve3d(c, prob3, phi, f, z, check=False)
        if r["rc"] != want or r["status"] != want or fake.fake_blocks() > 6: print(prec, r, fake.fake_blocks())
    ext.ext_destroy(c)
print(faults())
""")
    assert out.strip() == ""


def test_the_last_block_of_iterations_is_read(fake_cuda):
    """A solve that converges, or whose wait runs out, in the last block its limit allows reports that."""
    out = fake_cuda("""
phi, f, z = [Dev(128 ** 3) for _ in range(3)]
G, maxit = 10, 40
for prec, profile in (("fp32", 0), ("mixed_bf16", 0), ("mixed_bf16", 1)):
    c = ext.ext_create(ext.options(prec, maxit=maxit, iters_per_launch=G, profile=profile))
    prob = ext.problem(200, 150, "dirichlet")
    blocks = maxit // G + 8
    fake.fake_model(1, blocks, 0)
    r = ext.ext_solve(c, prob, phi, f, z, check=False)
    if (r["rc"], r["iters"]) != (0, blocks): print("2-D", prec, r)
    # the first product of the last block, after the first pass's four, a block's 4 G and its tail's 4
    fake.fake_model(1, 0, 4 + (blocks - 1) * 4 * (G + 1) + 1)
    r = ext.ext_solve(c, prob, phi, f, z, check=False)
    if r["rc"] != ext.EXT_ETIMEOUT: print("2-D flag", prec, r)
    fake.fake_model(1, 2, 0)
    r = ext.ext_solve(c, prob, phi, f, z, check=False)
    if (r["rc"], r["iters"]) != (0, 2): print("2-D after a time-out", prec, r)
    ext.ext_destroy(c)
c = ext.ext_create(ext.options("fp32", maxit=64))
fake.fake_model(1, 25, 0)
r = ext.ext_solve3d(c, ext.problem3(12, 12, 12), phi, f, z, check=False)
if (r["rc"], r["iters"]) != (0, 25): print("3-D", r)
ext.ext_destroy(c)
print(faults())
""")
    assert out.strip() == ""


def test_a_3d_solve_that_stagnates_runs_to_its_iteration_limit(fake_cuda):
    """One iteration a block, as when the recursive residual converges again and again and the true one does
    not: the solve ends as not converged at maxit."""
    out = fake_cuda("""
phi, f, z = [Dev(12 ** 3) for _ in range(3)]
for maxit in (1, 8, 64, 333):
    c = ext.ext_create(ext.options("fp32", maxit=maxit))
    fake.fake_model(1, 0, 0)
    r = ext.ext_solve3d(c, ext.problem3(12, 12, 12), phi, f, z, check=False)
    if (r["rc"], r["status"], r["iters"]) != (ext.EXT_ENOTCONV, ext.EXT_ENOTCONV, maxit): print(maxit, r)
    ext.ext_destroy(c)
""")
    assert out.strip() == ""


def test_3d_residual_replacements_come_when_they_are_due(fake_cuda):
    """The 3-D solve replaces its residual at the iteration that calls for it: a fall by replace_factor
    since the last replacement, true_res_every iterations since then, or the recursive residual's
    convergence, whatever the length of the blocks that it enqueues.  The residuals are given, the
    decisions the library's own; the rule is restated here."""
    out = fake_cuda("""
phi, f, z = [Dev(12 ** 3) for _ in range(3)]
rng = np.random.default_rng(1)
for every, factor, fall in itertools.product((1, 5, 11, 200), (1e-1, 1e-2), (0.25, 0.7)):
    rr = np.cumprod(fall * np.exp(0.8 * rng.standard_normal(400)))
    want, ref, since = [], 1.0, 0
    for it, v in enumerate(rr, 1):
        since += 1
        if v <= 1e-16 or v < factor ** 2 * ref or since >= every:
            want.append(it)
            ref, since = v * 1.0001, 0
            if v * 1.0001 <= 1e-16: break
    c = ext.ext_create(ext.options("fp32", maxit=400, iters_per_launch=1, true_res_every=every, replace_factor=factor))
    fake.fake_residuals(rr.ctypes.data_as(C.POINTER(C.c_double)), len(rr))
    r = ext.ext_solve3d(c, ext.problem3(12, 12, 12), phi, f, z, check=False)
    got = (C.c_int * 400)()
    n = fake.fake_replaced(got, 400)
    if list(got[:n]) != want or r["iters"] != want[-1] or r["rc"] != 0:
        print(every, factor, fall, list(got[:n]), want, r)
    ext.ext_destroy(c)
print(faults())
""")
    assert out.strip() == ""


@pytest.mark.parametrize("maxit", [400, 7])
def test_3d_result_tells_both_residuals(fake_cuda, maxit):
    """relres_rec is the recursive residual of the last iteration, relres_true the one recomputed."""
    out = fake_cuda("""
phi, f, z = [Dev(12 ** 3) for _ in range(3)]
rr = 0.3 ** np.arange(1, 100)
c = ext.ext_create(ext.options("fp32", maxit=%d))
fake.fake_residuals(rr.ctypes.data_as(C.POINTER(C.c_double)), len(rr))
r = ext.ext_solve3d(c, ext.problem3(12, 12, 12), phi, f, z, check=False)
v = rr[r["iters"] - 1]
assert r["iters"] > 5
if abs(r["relres_rec"] ** 2 / v - 1) > 1e-12 or abs(r["relres_true"] ** 2 / (v * 1.0001) - 1) > 1e-12: print(r, v)
""" % maxit)
    assert out.strip() == ""


def _footprint_before(nx, ny, six, low, host):
    """Bytes of a request's arena while FP32 mode kept double-float transform operands and the mixed modes
    four slices in four arrays: what a serving budget was set by."""
    pad = lambda n: (n + 127) // 128 * 128
    pays = lambda n: 2 * pad((n + 1) // 2) <= pad(n)
    off = [0]

    def take(b):
        off[0] = (off[0] + int(b) + 255) // 256 * 256
    n, nxp, nyp = nx * ny, pad(nx), pad(ny)
    fx, fy = pays(nx), pays(ny)
    hx, hy = (nx + 1) // 2 if fx else nx, (ny + 1) // 2 if fy else ny
    gm = (nxp // 128) * (nyp // 64)
    unfold = -(-hx // 32) * -(-hy // 8) if fx or fy else 0
    parts = max(-(-nx // 64) * -(-ny // 32), -(-n // 4096), gm, unfold)
    for b in (8 * n, 4 * n, 4 * n, 32 * parts, 8 * -(-ny // 16) * -(-nx // 32), *[4 * n] * 5, n, *[4 * n] * 5):
        take(b)
    for _ in range(6):
        take(0 if not six or fx or fy else 4 * nxp * nyp)
    take(4 * nxp), take(4 * nyp)
    if host:
        take(12 * n)
    if nx % 16 == 0:
        take(7 * 128)
    if not six or fx or fy:
        cx, cy = pad(hx), pad(hy)
        for _ in range((2 if fx else 1) * (2 if fy else 1)):
            if six:
                for _ in range(3):
                    take(8 * cx * cy)
                take(8 * hx * hy)
            else:
                take(2 * (6 if low else 4) * cx * cy)
                for _ in range(3):
                    take(8 * cx * cy)
                take(8 * 128), take(cx * cy // 16)
            if fx or fy:
                take(4 * cx), take(4 * cy), take(8 * hx * hy)
            if low:
                take(8 * 32 * 32 * (cy // 128)), take(12 * cx * 32), take(cx), take(8 * hx * hy), take(4 * 128)
    return off[0]


@pytest.mark.parametrize("prec,low", [("fp32", 2), ("mixed_bf16", 2), ("mixed_fp16", 1)])
def test_a_budget_admits_what_it_admitted(fake_cuda, prec, low):
    """A request is admitted at the footprint it had with the operands of before: axes that fold and do not, rows of tensor copies and not, host and device arrays."""
    shapes = [(4, 4), (64, 64), (130, 140), (127, 300), (389, 251), (512, 512), (1024, 700), (300, 2048)]
    budgets = [(nx, ny, host, _footprint_before(nx, ny, prec == "fp32", prec != "fp32" and (low == 1 or ny >= 2048), host))
               for nx, ny in shapes for host in (False, True)]
    out = fake_cuda("""
for nx, ny, host, budget in %r:
    arrays = [np.zeros((ny, nx), np.float32) if host else Dev(nx * ny) for _ in range(3)]
    c = ext.ext_create(ext.options(%r, low_modes=%d, hbm_budget=budget))
    fake.fake_model(5, 1, 0)
    t = ext.ext_submit(c, ext.problem(nx, ny, "dirichlet"), *arrays)
    ext.ext_drain(c)
    r = ext.ext_poll(c, t)["rc"]
    if r != 0: print(nx, ny, host, budget, r)
    ext.ext_destroy(c)
print(faults())
""" % (budgets, prec, low))
    assert out.strip() == ""


def test_profiled_graphs_own_their_events(fake_cuda):
    """A serving table whose mixes of requests need several iteration graphs, and solves that capture again
    after a change of the tile height: every event made is destroyed with the context."""
    out = fake_cuda("""
phi, f, out = [Dev(300 * 300) for _ in range(3)]
before = fake.fake_events()
c = ext.ext_create(ext.options("mixed_bf16", profile=1, low_modes=2))
for shape in ((60, 60), (300, 290), (250, 200), (60, 60)):  # unfolded, partly folded, folded
    fake.fake_model(5, 2, 0)
    t = ext.ext_submit(c, ext.problem(*shape, "dirichlet"), phi, f, out)
    ext.ext_drain(c)
    if ext.ext_poll(c, t)["rc"] != 0: print(shape)
    fake.fake_model(5, 2, 0)
    r = ext.ext_solve(c, ext.problem(*shape, "dirichlet"), phi, f, out, check=False)
    if r["rc"] != 0: print(shape, r)
# each solve's two blocks of ten iterations are in the totals
if ext.ext_profile_read(c)["true_residual"][1] != 8: print(ext.ext_profile_read(c))
ext.ext_destroy(c)
if fake.fake_events() != before: print(fake.fake_events() - before, "events left")
""")
    assert out.strip() == ""


def test_creating_a_context_waits_for_no_work_of_the_caller(fake_cuda):
    """The caller's default stream may be busy with the inputs of the next call."""
    out = fake_cuda("""
before = fake.fake_legacy_waits()
c = ext.ext_create(ext.options("mixed_bf16"))
if fake.fake_legacy_waits() != before: print(fake.fake_legacy_waits() - before)
print(faults())
""")
    assert out.strip() == ""
