"""The FP32 path's workspace: vectors for passes of 8 RHS are asked for after everything else
that an operator needs, and an operator that does not get them applies 4 RHS a pass."""
import numpy as np
import pytest

from mbf_synth import complex_normal

from gpu_util import gpu_apply, import_factors, oracle_case, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_SIMT = 1e-5


def test_wide_vectors_are_the_last_allocation_and_can_be_done_without():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_07925_gb300 import binding as bd
    from paper_1509_07925_gb300 import buildlib
    buildlib.build()
    fs, sb = oracle_case("fio_iso", 64, 2, 4, 24, "polar")
    hf = import_factors(bd, fs)
    g = complex_normal(fs.n_in, 13, seed=35).astype(np.complex64).astype(np.complex128)
    v = complex_normal(fs.n_out, 13, seed=36).astype(np.complex64).astype(np.complex128)
    ref, refa = sb.apply(g), sb.adjoint(v)
    outcome = []          # of a creation whose k-th allocation fails: refused, lesser, narrow or whole
    try:
        for k in range(40):
            bd._check(bd.lib().mbf_debug_fail_alloc(k))
            try:
                op = bd.Operator(hf)
            except bd.MbfError as e:
                assert e.code == bd.MBF_ERR_OOM
                outcome.append("refused")
                continue
            bd._check(bd.lib().mbf_debug_fail_alloc(-1))
            whole = bool(op.info().tensor_ok)
            if whole:
                op.set_profiling(True)
                gpu_apply(torch, op, g[:8], precision=bd.MBF_PREC_FP32_SIMT)
                passes = op.profile()["bf_apply_simt"][0]
                assert passes in (1, 2)
                outcome.append("whole" if passes == 1 else "narrow")
                if passes == 2:                       # passes of 4, 4, 4 and 1 RHS
                    for adjoint, x, r in ((False, g, ref), (True, v, refa)):
                        for nrhs in (5, 13):
                            u = gpu_apply(torch, op, x[:nrhs], adjoint=adjoint, precision=bd.MBF_PREC_FP32_SIMT)
                            assert max(rel(u[j], r[j]) for j in range(nrhs)) <= TOL_SIMT
            else:
                outcome.append("lesser")
            op.close()
    finally:
        bd._check(bd.lib().mbf_debug_fail_alloc(-1))
    assert outcome.count("narrow") == 1 and outcome[-1] == "whole"
    at = outcome.index("narrow")
    # nothing that the operator cannot do without comes behind it (the creation makes at + 1 allocations)
    assert all(o == "whole" for o in outcome[at + 1:]) and "refused" in outcome[:at] and "lesser" in outcome[:at]
