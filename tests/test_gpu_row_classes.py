"""Alias rows on both sides of every class bound of the row kernel (rows of up to 512 slots, of up
to 1200, longer; tasks of all classes in one build) against their own weights, and the inelastic
and thermal walks over walker counts around their warps' chunks: a tally of N walkers is the sum
of the tallies of its two parts (counter-based draws: a walker's walk depends on its id alone).
Bars: (K + 2) 2^-32 per outcome (quantisation of an exact integer row), counts equal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import alias  # noqa: E402
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


def _wire(W, L, n_energy=1):
    return inputs.small_wire(700 + W + L, W, L, n_energy=n_energy, eta=0.06, disorder=0.8,
                             e_lo=0.2, e_hi=0.5)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("sizes", [((1, 1),), ((10, 51),), ((7, 73),), ((2, 599),), ((11, 109),),
                                   ((1, 30), (1, 31), (10, 51), (7, 73), (2, 599), (11, 109))],
                         ids=["K3", "K512", "K513", "K1200", "K1201", "all"])
def test_rows_of_every_class(ctx, sizes, precision):
    wires = [_wire(W, L) for W, L in sizes]
    tables = negf.negf_build_tables(ctx, wires, precision=precision, keep_weights=True,
                                    layout="one_level")
    try:
        for task, (W, L) in enumerate(sizes):
            rows, K = W * L + 2 * W, W * L + 2
            w = negf.negf_export_tables(ctx, tables, task, "weights").reshape(rows, K)
            rs = negf.negf_export_tables(ctx, tables, task, "rowsum")
            ent = negf.negf_export_tables(ctx, tables, task, "alias").reshape(rows, K)
            for r in sorted({0, 1, rows // 3, W * L - 1, W * L, rows - 1}):
                if rs[r] <= 0:
                    continue
                p = alias.implied_distribution(ent[r])
                assert np.max(np.abs(p - w[r] / rs[r])) <= (K + 2) / 2**32 + 1e-12, (W, L, r)
    finally:
        negf.negf_tables_free(tables)


def _inelastic(ctx, tables, nE, N, off):
    tally = negf.negf_walk_inelastic(ctx, tables, 0, 31, N, 0.3, walker_id_offset=off)
    try:
        return negf.negf_tally_counts(ctx, tally, nE)
    finally:
        negf.negf_tally_free(tally)


@pytest.mark.parametrize("N", [2, 31, 33, 513, 40_961, 1_000_003])
def test_chunked_walks_add_up(ctx, N):
    nE = 5
    tables = negf.negf_build_tables(ctx, [_wire(3, 9, nE)], precision="fp32")
    try:
        h = N // 3 + 1
        whole = _inelastic(ctx, tables, nE, N, 7)
        assert np.array_equal(whole, _inelastic(ctx, tables, nE, h, 7)
                              + _inelastic(ctx, tables, nE, N - h, 7 + h))
        assert np.all(whole[:, 0] == N)
        t = [negf.negf_walk_thermal(ctx, tables, 0, 0, 32, n, 0.35, 0.03, walker_id_offset=off)
             for n, off in ((N, 7), (h, 7), (N - h, 7 + h))]
        assert t[0]["walkers"] == N
        for q in (0, 1):
            assert t[0]["absorbed"][q] == t[1]["absorbed"][q] + t[2]["absorbed"][q]
        steps = [x["mean_steps"] * x["walkers"] for x in t]
        assert abs(steps[0] - steps[1] - steps[2]) <= 1e-9 * steps[0]
    finally:
        negf.negf_tables_free(tables)
