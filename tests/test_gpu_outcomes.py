"""What the calls tell their callers, and results at the ends of FP32's range (GB300)."""

import numpy as np
import pytest

from oracle import biharmonic as ob

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
