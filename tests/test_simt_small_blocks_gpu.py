"""GPU parity of the FP32 SIMT kernel on blocks smaller than a warp's lanes: rows of 4 to 64
entries, so that up to 32 lines go side by side in a warp (2-D and 3-D, counts that are
no power of two among them), leaves of a single point and rank, and groups with no
lines at all, against the oracle's FP64 apply of the library's factors."""
import numpy as np
import pytest

from mbf_synth import complex_normal
from oracle import bf as B
from paper_1509_07925_gb300.binding import MBF_PREC_FP32_SIMT, MBF_TREE_POLAR, MBF_TREE_UNIFORM

from gpu_util import export_factors, gpu_apply, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_SIMT = 1e-5


@pytest.mark.parametrize("dim,n,L,r,tree", [
    (2, 16, 4, 1, MBF_TREE_UNIFORM),    # rows of 4: 32 lines side by side
    (2, 16, 4, 3, MBF_TREE_UNIFORM),    # rows of 12 (and 4 at the leaves): 10 lines
    (2, 32, 4, 5, MBF_TREE_UNIFORM),    # rows of 20 and 16: 6 and 8 lines
    (2, 64, 6, 7, MBF_TREE_UNIFORM),    # 1024 groups, two CTAs to an SM; rows of 28: 4 lines
    (2, 64, 6, 11, MBF_TREE_POLAR),     # rows of 44: 2 lines; empty leaves
    (3, 8, 2, 3, MBF_TREE_UNIFORM),     # rows of 24: 5 lines, eight segments
])
def test_small_blocks_match_oracle(dim, n, L, r, tree):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_07925_gb300 import binding as bd
    from paper_1509_07925_gb300 import buildlib
    buildlib.build()
    hf = bd.HostFactors.build(dim, n, L, r, tree=tree, kernel="fio_iso" if tree == MBF_TREE_POLAR else "dft")
    op, sb = bd.Operator(hf), B.SparseBF(export_factors(hf.arrays()))
    g = complex_normal(n ** dim, 5, seed=43).astype(np.complex64).astype(np.complex128)
    for adjoint in (False, True):
        ref = sb.adjoint(g) if adjoint else sb.apply(g)
        for nrhs in (1, 2, 5):
            u = gpu_apply(torch, op, g[:nrhs], adjoint=adjoint, precision=MBF_PREC_FP32_SIMT)
            for k in range(nrhs):
                assert rel(u[k], ref[k]) <= TOL_SIMT, (adjoint, nrhs, k, rel(u[k], ref[k]))
    op.close()
