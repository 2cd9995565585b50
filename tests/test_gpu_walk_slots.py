"""Two-level walks at one and at two walkers per lane: a launch of many walkers (one per lane at a
time) counts what its parts count (two), task by task; narrow slices (always one) the same."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1805_10164_gb300 import inputs, negf  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_10164_gb300 import build
    build.build()
    c = negf.negf_create(0)
    yield c
    negf.negf_destroy(c)


def _counts(ctx, tables, n, N, off):
    tally = negf.negf_walk(ctx, tables, 1, 91, N, walker_id_offset=off)
    try:
        return negf.negf_tally_counts(ctx, tally, n)
    finally:
        negf.negf_tally_free(tally)


@pytest.mark.parametrize("W,L", [(4, 9), (5, 7), (17, 3)])
def test_many_walkers_count_what_their_parts_count(ctx, W, L):
    n = 5
    w = inputs.small_wire(660 + W, W, L, n_energy=n, eta=0.1, e_lo=-1.9, e_hi=1.7)
    tables = negf.negf_build_tables(ctx, [w], precision="fp32", layout="two_level")
    try:
        lanes = 4 * 256 * torch.cuda.get_device_properties(0).multi_processor_count
        N = 45 * lanes // n + 3
        h = N // 2 + 11
        whole = _counts(ctx, tables, n, N, 2 ** 32 - 50)
        assert np.array_equal(whole, _counts(ctx, tables, n, h, 2 ** 32 - 50)
                              + _counts(ctx, tables, n, N - h, 2 ** 32 - 50 + h))
        assert np.all(whole[:, 0] == N)
    finally:
        negf.negf_tables_free(tables)
