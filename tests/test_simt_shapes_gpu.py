"""GPU parity of the FP32 SIMT kernel over the shapes its work split depends on: every RHS
count of a pass (1, 2, 4, 8, padded ones, several passes), one and two CTAs to an SM
(fewer and more groups than two per SM), entries split over lanes and warps (rows of 20
to 256), blocks longer than the chunk ring, 2-D and 3-D, forward and adjoint, against
the oracle's FP64 apply of the library's factors."""
import functools

import numpy as np
import pytest

from mbf_synth import complex_normal
from oracle import bf as B
from paper_1509_07925_gb300.binding import MBF_PREC_FP32_SIMT, MBF_TREE_POLAR, MBF_TREE_UNIFORM

from gpu_util import export_factors, gpu_apply, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_SIMT = 1e-5

CASES = [
    # dim, n, L, r, tree, kernel
    (2, 16, 2, 5, MBF_TREE_UNIFORM, "dft"),       # 4 groups, rows of 20
    (2, 32, 2, 33, MBF_TREE_UNIFORM, "dft"),      # rows of 132: split over two sets of warps
    (2, 32, 2, 64, MBF_TREE_UNIFORM, "dft"),      # 256 x 256 blocks (86 chunks), 256-point groups
    (3, 8, 2, 27, MBF_TREE_UNIFORM, "dft"),       # 8 groups, rows of 216, eight leaves a group
    (3, 16, 4, 16, MBF_TREE_UNIFORM, "dft"),      # 512 groups: two CTAs to an SM, eight leaves
    (2, 64, 6, 9, MBF_TREE_POLAR, "fio_iso"),     # 1024 groups, ragged and empty leaves, odd rank
]


@pytest.fixture(scope="module")
def ops():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1509_07925_gb300 import buildlib
    buildlib.build()
    from paper_1509_07925_gb300 import binding as bd

    @functools.lru_cache(maxsize=None)
    def make(case):
        dim, n, L, r, tree, kernel = case
        hf = bd.HostFactors.build(dim, n, L, r, tree=tree, kernel=kernel)
        return bd.Operator(hf), B.SparseBF(export_factors(hf.arrays())), n ** dim
    return make


@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("case", CASES)
def test_simt_shapes_match_oracle(ops, case, adjoint):
    op, sb, points = ops(case)
    g = complex_normal(points, 13, seed=41).astype(np.complex64).astype(np.complex128)
    ref = sb.adjoint(g) if adjoint else sb.apply(g)
    for nrhs in (1, 2, 3, 4, 5, 8, 13):
        u = gpu_apply(torch, op, g[:nrhs], adjoint=adjoint, precision=MBF_PREC_FP32_SIMT)
        assert np.all(np.isfinite(u))
        for k in range(nrhs):
            assert rel(u[k], ref[k]) <= TOL_SIMT, (case, adjoint, nrhs, k, rel(u[k], ref[k]))
