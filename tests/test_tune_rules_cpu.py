"""The autotuner's rules as pure host functions: what it times (the configuration that the
operator has among it) and the RHS count from which AUTO takes the tensor cores."""
import pytest


@pytest.fixture(scope="module")
def bd():
    from paper_1509_07925_gb300 import binding, buildlib
    buildlib.build()
    return binding


def test_the_present_configuration_is_timed_first(bd):
    # one buffer and six slots, as creation chooses for tiles of 160 rows: kept unless beaten
    assert bd.tune_candidates(6, 1, [6, 2, 0]) == [(6, 1), (2, 2)]
    # two buffers and the deepest ring: as many candidates as ever, each once
    c = bd.tune_candidates(10, 2, [14, 10, 6])
    assert c[0] == (10, 2) and len(c) == len(set(c)) == 8
    assert set(c) == {(n, 2) for n in (2, 4, 6, 8, 10)} | {(n, 3) for n in (2, 4, 6)}
    # never more than 8, nor a ring deeper than what fits
    for cur in ((2, 1), (16, 2), (4, 3)):
        for deepest in ([16, 16, 16], [16, 12, 0], [8, 0, 0], [4, 2, 2]):
            c = bd.tune_candidates(*cur, deepest)
            assert c[0] == cur and 1 <= len(c) <= 8 and len(set(c)) == len(c)
            assert all(2 <= n <= deepest[b - 1] for n, b in c[1:])


def test_crossover_follows_the_panel_that_is_filled(bd):
    rhs, simt = [1, 2, 4, 8, 16, 32, 64], [0.08, 0.09, 0.11, 0.19, 0.37, 0.74, 1.5]
    assert bd.tune_crossover(rhs, simt, 0.10, 0.17) == 4       # a panel of 32 beats the SIMT apply here
    assert bd.tune_crossover(rhs, simt, 0.17, 0.17) == 8
    assert bd.tune_crossover(rhs, simt, 0.80, 1.0) == 64       # only a full panel does
    assert bd.tune_crossover(rhs, simt, 2.0, 2.0) == 65
    assert bd.tune_crossover([], [], 1.0, 1.0) == 65
