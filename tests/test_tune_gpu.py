"""The autotuner on tiles so wide that creation gives them one panel buffer and a deeper ring:
that configuration is among those timed, and the one kept is the fastest timed."""
import numpy as np
import pytest

from mbf_synth import complex_normal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_tuner_times_the_configuration_of_creation():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_07925_gb300 import binding as bd
    from paper_1509_07925_gb300 import buildlib
    buildlib.build()
    op = bd.Operator(bd.HostFactors.build(2, 32, 2, 40))       # tiles of 160 x 160
    slots = op.info().tensor_slots
    st = torch.cuda.current_stream().cuda_stream
    g = torch.from_numpy(complex_normal(32 * 32, 64, seed=91).astype(np.complex64)).cuda()
    ref, u = torch.empty_like(g), torch.empty_like(g)
    op.apply(g.data_ptr(), ref.data_ptr(), 64, bd.MBF_PREC_BF16X3, st)
    r = op.tune(st)
    tried = list(zip(r.slots, r.panel_buffers))[:r.n_slots]
    assert tried[0] == (slots, 1) and (2, 2) in tried
    best = min(range(r.n_slots), key=lambda k: r.tc_ms[k])
    assert (r.tc_slots_chosen, r.tc_buffers_chosen) == tried[best] and op.info().tensor_slots == tried[best][0]
    for nrhs in (64, 20):                                      # the same bits in any configuration
        op.apply(g.data_ptr(), u.data_ptr(), nrhs, bd.MBF_PREC_BF16X3, st)
        op.check(st)
        assert torch.equal(torch.view_as_real(u[:nrhs]), torch.view_as_real(ref[:nrhs])), nrhs
    op.close()
