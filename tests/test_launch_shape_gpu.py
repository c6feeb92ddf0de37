"""mbf_op_info reports the SIMT launch that is made: two CTAs to an SM where every one has a
group per stage, else one for each group up to one to an SM."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,L,groups", [(2, 16, 2, 4), (2, 64, 4, 64), (2, 64, 6, 1024), (3, 16, 4, 512)])
def test_reported_shape(dim, n, L, groups):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_07925_gb300 import binding as bd
    from paper_1509_07925_gb300 import buildlib
    buildlib.build()
    op = bd.Operator(bd.HostFactors.build(dim, n, L, 6))
    inf = op.info()
    p = torch.cuda.get_device_properties(0)
    sms, pair = p.multi_processor_count, groups >= 2 * p.multi_processor_count
    assert inf.grid == (2 * sms if pair else min(sms, groups))
    per_sm = 2 if pair else 1
    assert inf.threads * per_sm <= 1024 and inf.threads == (256 if pair else 448)
    assert 0 < inf.smem and per_sm * (inf.smem + 1024) <= p.shared_memory_per_multiprocessor
    op.close()
