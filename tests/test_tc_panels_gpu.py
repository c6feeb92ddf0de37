"""GPU parity of the tensor-core path's two panel widths: RHS counts that fill, leave room
in and span panels of 64 and of 32, forward (split-BF16x3 and TF32) and adjoint, on
stacked and wide tiles, 2-D and 3-D, against the oracle's FP64 apply of the same factors;
and the multiscale sum with a panel of 32 (accumulating parts)."""
import numpy as np
import pytest

from mbf_synth import complex_normal
from oracle import msbf as MS
from oracle import problem as P
from paper_1509_07925_gb300.binding import MBF_PREC_BF16X3, MBF_PREC_TF32

from gpu_util import gpu_apply, import_factors, oracle_case, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_BF16X3 = 1e-4
TOL_TF32 = 5e-3

CASES = [
    ("dft", 16, 2, 2, 5, "none"),         # rank rounded up to 8, leaf blocks of 32 threads
    ("fio_iso", 64, 2, 4, 24, "polar"),   # ragged and empty leaves (up to 38 points)
    ("dft", 8, 3, 2, 16, "none"),         # c = 8, 128-row tiles
    ("dft", 32, 2, 2, 64, "none"),        # 256-row tiles: one plane an MMA, one panel buffer
]


@pytest.fixture(scope="module")
def bd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_07925_gb300 import buildlib
    buildlib.build()
    from paper_1509_07925_gb300 import binding
    return binding


@pytest.mark.parametrize("case", CASES)
def test_panels_match_oracle(bd, case):
    fs, sb = oracle_case(*case)
    op = bd.Operator(import_factors(bd, fs))
    g = complex_normal(fs.n_in, 96, seed=51).astype(np.complex64).astype(np.complex128)
    w = complex_normal(fs.n_out, 96, seed=52).astype(np.complex64).astype(np.complex128)
    ref, refa = sb.apply(g), sb.adjoint(w)
    for nrhs in (9, 32, 33, 96):
        for prec, tol in ((MBF_PREC_BF16X3, TOL_BF16X3), (MBF_PREC_TF32, TOL_TF32)):
            u = gpu_apply(torch, op, g[:nrhs], precision=prec)
            assert max(rel(u[k], ref[k]) for k in range(nrhs)) <= tol, (case, nrhs, prec)
        v = gpu_apply(torch, op, w[:nrhs], adjoint=True, precision=MBF_PREC_BF16X3)
        assert max(rel(v[k], refa[k]) for k in range(nrhs)) <= TOL_BF16X3, (case, nrhs)
    op.close()


@pytest.mark.parametrize("nrhs", [13, 40])
def test_multiscale_sum_with_narrow_panels(bd, nrhs):
    n, r, nc = 32, 8, 8
    m = MS.build(P.kernel_fio_iso, n, r, n_center=nc)
    sm = MS.SparseMsBF(m)
    gm = bd.MsBF.create([bd.Operator(import_factors(bd, fs)) for _, _, _, fs in m.parts], m.Kc.T, m.center)
    st = torch.cuda.current_stream().cuda_stream
    for adjoint in (False, True):
        g = complex_normal(n * n, nrhs, seed=53)
        gt = torch.from_numpy(g.astype(np.complex64)).cuda()
        ut = torch.full((nrhs, n * n), float("nan"), dtype=torch.complex64, device="cuda")
        (gm.apply_adjoint if adjoint else gm.apply)(gt.data_ptr(), ut.data_ptr(), nrhs, MBF_PREC_BF16X3, st)
        gm.check(st)
        ref = sm.adjoint(g) if adjoint else sm.apply(g)
        u = ut.cpu().numpy()
        assert max(rel(u[k], ref[k]) for k in range(nrhs)) <= TOL_BF16X3, (nrhs, adjoint)
    gm.close()


def test_small_sm_share_ends_without_a_wait_running_out(bd):
    """1024 groups per level on the few SMs of a served batch's share: over a hundred groups
    a CTA and level, so that every role of the kernel may run many groups ahead of another;
    no request takes anywhere near the 2 s after which a device wait gives up."""
    import time
    hf = bd.HostFactors.build(2, 64, 6, 8)
    op = bd.Operator(hf)
    g = torch.from_numpy(complex_normal(64 * 64, 64, seed=61).astype(np.complex64)).cuda()
    ref = torch.empty_like(g)
    st = torch.cuda.current_stream().cuda_stream
    op.apply(g.data_ptr(), ref.data_ptr(), 64, MBF_PREC_BF16X3, st)
    op.check(st)
    srv = bd.Server(staging_budget_bytes=1 << 28, max_inflight=16, max_batch_rhs=64)
    outs = [torch.zeros_like(g) for _ in range(48)]
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for k, u in enumerate(outs):
        srv.submit(op, g.data_ptr(), u.data_ptr(), 64 if k % 2 else 20)
    srv.drain(30.0)
    elapsed = time.perf_counter() - t0
    srv.close()
    assert elapsed < 1.0, elapsed
    for k, u in enumerate(outs):
        n = 64 if k % 2 else 20
        assert torch.linalg.norm(u[:n] - ref[:n]) <= 2e-4 * torch.linalg.norm(ref[:n])
    op.close()
