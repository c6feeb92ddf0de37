"""Applies of one operator captured in one CUDA graph and replayed: forward and adjoint, FP32
and tensor cores, all over the operator's own workspace.  The kernels' dependency
counters come in two sets that the launches flip on the device, so a replay may start
with either, after any number of launches outside the graph."""
import numpy as np
import pytest

from mbf_synth import complex_normal
from paper_1509_07925_gb300.binding import MBF_PREC_BF16X3, MBF_PREC_FP32_SIMT, MBF_PREC_TF32

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

APPLIES = [(5, MBF_PREC_FP32_SIMT, False), (64, MBF_PREC_BF16X3, False), (3, MBF_PREC_FP32_SIMT, True),
           (32, MBF_PREC_BF16X3, True), (20, MBF_PREC_TF32, False)]


@pytest.mark.parametrize("n,L", [(32, 4), (64, 6)])      # one and two SIMT CTAs to an SM
def test_replays_equal_eager_applies(n, L):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_07925_gb300 import binding as bd
    from paper_1509_07925_gb300 import buildlib
    buildlib.build()
    op = bd.Operator(bd.HostFactors.build(2, n, L, 8))
    ins = [torch.empty(nrhs, n * n, dtype=torch.complex64, device="cuda") for nrhs, _, _ in APPLIES]
    outs = [torch.empty_like(x) for x in ins]

    def fill(seed):
        for k, x in enumerate(ins):
            x.copy_(torch.from_numpy(complex_normal(n * n, x.shape[0], seed=seed + k).astype(np.complex64)))

    def run():
        st = torch.cuda.current_stream().cuda_stream
        for (nrhs, prec, adjoint), x, y in zip(APPLIES, ins, outs):
            (op.apply_adjoint if adjoint else op.apply)(x.data_ptr(), y.data_ptr(), nrhs, prec, st)

    fill(1)
    run()                                                 # workspaces and tiles made before the capture
    op.check(torch.cuda.current_stream().cuda_stream)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    st = torch.cuda.current_stream().cuda_stream
    for i in range(6):
        fill(100 * (i + 2))
        run()
        if i % 2:                                         # an odd number of launches between replays
            op.apply(ins[0].data_ptr(), outs[0].data_ptr(), 1, MBF_PREC_FP32_SIMT, st)
            op.apply(ins[1].data_ptr(), outs[1].data_ptr(), 9, MBF_PREC_BF16X3, st)
            run()
        op.check(st)
        ref = [y.clone() for y in outs]
        for y in outs:
            y.fill_(float("nan"))
        graph.replay()
        graph.replay()
        op.check(st)
        for k, (y, r) in enumerate(zip(outs, ref)):
            assert torch.equal(torch.view_as_real(y), torch.view_as_real(r)), (i, k)
    op.close()
