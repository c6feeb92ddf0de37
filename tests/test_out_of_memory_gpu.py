"""Device allocations that the device refuses: the call reports MBF_ERR_OOM and nothing else
is affected by it.  The refused one is a staging buffer larger than any device's memory
(2^24 RHS of 4096 points, 549 GB), asked for before any byte is copied."""
import ctypes as C

import numpy as np
import pytest

from mbf_synth import complex_normal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, HUGE = 64, 1 << 24


@pytest.fixture()
def bd_op():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_07925_gb300 import binding as bd
    from paper_1509_07925_gb300 import buildlib
    buildlib.build()
    op = bd.Operator(bd.HostFactors.build(2, N, 4, 8))
    yield bd, op
    op.close()


def _refused(bd, op):
    h = np.zeros(16, np.complex64)      # (never read)
    p = h.ctypes.data_as(C.c_void_p)
    with pytest.raises(bd.MbfError) as e:
        bd._check(bd.lib().mbf_apply_host(op._h, p, p, HUGE, bd.MBF_PREC_FP32_SIMT, None))
    assert e.value.code == bd.MBF_ERR_OOM, str(e.value)


def test_a_refused_allocation_leaves_no_error_behind(bd_op):
    """A later check of the CUDA runtime's last error, as launches are followed by, must not
    find the refusal, which the call has reported."""
    bd, op = bd_op
    cudart = C.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    g = torch.from_numpy(complex_normal(N * N, 64, seed=81).astype(np.complex64)).cuda()
    out = [torch.zeros_like(g) for _ in range(2)]
    st = torch.cuda.current_stream().cuda_stream
    op.apply(g.data_ptr(), out[0].data_ptr(), 64, bd.MBF_PREC_BF16X3, st)
    _refused(bd, op)
    assert cudart.cudaPeekAtLastError() == 0
    op.apply(g.data_ptr(), out[1].data_ptr(), 64, bd.MBF_PREC_BF16X3, st)
    op.check(st)
    assert torch.equal(torch.view_as_real(out[0]), torch.view_as_real(out[1]))


def test_staging_is_allocated_again_after_a_refusal(bd_op):
    """The refused larger staging buffer took the place of the one there was."""
    bd, op = bd_op
    g = complex_normal(N * N, 2, seed=82).astype(np.complex64)
    ref = op.apply_host(g, 2, bd.MBF_PREC_FP32_SIMT)
    _refused(bd, op)
    assert np.array_equal(op.apply_host(g, 2, bd.MBF_PREC_FP32_SIMT), ref)
