"""The tensor kernel's hand-over of stage vectors between CTAs under repetition: applies of
two inputs in turn over one workspace, so that every block still holds the other input's
values until its producer has written it, give the same bits each time."""
import pytest

from mbf_synth import complex_normal
from paper_1509_07925_gb300.binding import MBF_PREC_BF16X3, MBF_PREC_TF32

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs,precision,adjoint", [(64, MBF_PREC_BF16X3, False), (20, MBF_PREC_BF16X3, False),
                                                    (64, MBF_PREC_TF32, False), (32, MBF_PREC_BF16X3, True)])
def test_repeated_applies_give_the_same_bits(nrhs, precision, adjoint):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_07925_gb300 import binding as bd
    from paper_1509_07925_gb300 import buildlib
    buildlib.build()
    op = bd.Operator(bd.HostFactors.build(2, 64, 6, 8))     # 1024 groups a level
    st = torch.cuda.current_stream().cuda_stream
    ins = [torch.from_numpy(complex_normal(64 * 64, nrhs, seed=s).astype("complex64")).cuda() for s in (71, 72)]
    apply = op.apply_adjoint if adjoint else op.apply

    def run(k):
        out = torch.full_like(ins[k], float("nan"))
        apply(ins[k].data_ptr(), out.data_ptr(), nrhs, precision, st)
        return out

    ref = [run(0), run(1)]
    op.check(st)
    assert not torch.equal(ref[0], ref[1])
    for i in range(200):
        assert torch.equal(torch.view_as_real(run(i % 2)), torch.view_as_real(ref[i % 2])), i
    op.check(st)
    op.close()
