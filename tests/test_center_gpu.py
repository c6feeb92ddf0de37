"""GPU parity of the dense centre term of the multiscale sum: point counts at the edges of a
staged round (512) and of the adjoint's sets of points, few RHS and so many that the
forward kernel changes its mapping, against the FP64 product with a random kernel."""
import numpy as np
import pytest

from mbf_synth import complex_normal

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 64
TOL = 1e-5      # FP32 sums of at most 4096 terms: some sqrt(4096) 6e-8


@pytest.fixture(scope="module")
def part():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_07925_gb300 import binding as bd
    from paper_1509_07925_gb300 import buildlib
    buildlib.build()
    return bd, bd.HostFactors.build(2, N, 4, 4)


@pytest.mark.parametrize("n_c", [1, 3, 4, 5, 290, 511, 512, 513])
def test_centre_matches_fp64(part, n_c):
    bd, hf = part
    op = bd.Operator(hf)
    rng = np.random.default_rng(n_c)
    centre = rng.permutation(N * N)[:n_c]
    K = complex_normal(N * N, n_c, seed=101)                   # [n_c][points]
    ms = bd.MsBF.create([bd.Operator(hf)], K, centre)
    st = torch.cuda.current_stream().cuda_stream
    Kd = torch.from_numpy(K).cuda()
    ci = torch.from_numpy(centre).cuda()
    for nrhs in (1, 9, 40, 160):                               # 160: 320 CTAs of 256 outputs and 8 RHS
        x = torch.from_numpy(complex_normal(N * N, nrhs, seed=nrhs).astype(np.complex64)).cuda()
        for adjoint in (False, True):
            y, z = torch.full_like(x, float("nan")), torch.zeros_like(x)
            (ms.apply_adjoint if adjoint else ms.apply)(x.data_ptr(), y.data_ptr(), nrhs, bd.MBF_PREC_FP32_SIMT, st)
            (op.apply_adjoint if adjoint else op.apply)(x.data_ptr(), z.data_ptr(), nrhs, bd.MBF_PREC_FP32_SIMT, st)
            ms.check(st)
            op.check(st)
            ref, x64 = z.to(torch.complex128), x.to(torch.complex128)
            if adjoint:
                ref[:, ci] += x64 @ Kd.conj().T
            else:
                ref += x64[:, ci] @ Kd
            err = torch.linalg.norm(y - ref, dim=1) / torch.linalg.norm(ref, dim=1)
            assert float(err.max()) <= TOL, (nrhs, adjoint, float(err.max()))
    ms.close()
    op.close()
