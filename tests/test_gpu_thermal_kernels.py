"""The two kernels of negf_walk_thermal walk alike: launches of more than three walkers a lane
(intervals staged in shared memory) against launches of their parts (few walkers: intervals read
where they are set up), walker by walker; and grids around the largest that is staged (652
energies) with many walkers, a sample of whose walks is replayed by the oracle.  A walker's
walk depends on its id alone, so everything is equal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import thermal  # noqa: E402
from paper_1805_10164_gb300 import inputs, negf  # noqa: E402

MU, KT = 0.1, 0.09


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_10164_gb300 import build
    build.build()
    c = negf.negf_create(0)
    yield c
    negf.negf_destroy(c)


def _many():
    """Walkers of a launch that the staging kernel takes."""
    return 3 * 4 * 256 * torch.cuda.get_device_properties(0).multi_processor_count + 1


def _tables(ctx, W, L, M, layout):
    w = inputs.small_wire(620 + W, W, L, n_energy=1, eta=0.1, disorder=0.8)
    w.energy = np.linspace(-0.3, 0.5, M)
    w.energy_weight = np.ones(M)
    return w, negf.negf_build_tables(ctx, [w], precision="fp32", layout=layout)


def _walk(ctx, tables, N, off):
    tr = {k: torch.empty(N, dtype=torch.int32, device="cuda")
          for k in ("lead", "steps", "interval", "a")}
    res = negf.negf_walk_thermal(ctx, tables, 0, 0, 77, N, MU, KT, walker_id_offset=off, trace=tr)
    return res, {k: t.cpu().numpy() for k, t in tr.items()}


@pytest.mark.parametrize("layout", ["one_level", "two_level"])
@pytest.mark.parametrize("W,L,M", [(3, 5, 2), (9, 7, 40)])
def test_parts_equal_whole(ctx, W, L, M, layout):
    _, tables = _tables(ctx, W, L, M, layout)
    try:
        N = _many() + 12
        h = N // 2 + 5
        res, tr = _walk(ctx, tables, N, 2 ** 33 - 100)
        parts = [_walk(ctx, tables, n, 2 ** 33 - 100 + o) for n, o in ((h, 0), (N - h, h))]
        for k in tr:
            assert np.array_equal(tr[k], np.concatenate([p[1][k] for p in parts])), k
        for q in (0, 1):
            assert res["absorbed"][q] == sum(p[0]["absorbed"][q] for p in parts)
            assert res["absorbed"][q] == np.count_nonzero(tr["lead"] == q)
        assert res["closed"] == sum(p[0]["closed"] for p in parts)
        # G N and the integer sums behind it add up
        G = sum(p[0]["G"] * n for p, n in zip(parts, (h, N - h)))
        assert abs(res["G"] * N - G) <= 1e-9 * abs(G)
    finally:
        negf.negf_tables_free(tables)


@pytest.mark.parametrize("layout", ["one_level", "two_level"])
@pytest.mark.parametrize("M", [652, 653, 1400])
def test_large_grids(ctx, M, layout):
    W, L = 2, 3
    w, tables = _tables(ctx, W, L, M, layout)
    try:
        res, tr = _walk(ctx, tables, _many(), 5)
        pick = np.sort(np.random.default_rng(M).choice(_many(), 1500, replace=False))
        ent, ment, c, l2 = [], [], [], []
        for e in range(M):
            info = negf.negf_get_task_info(ctx, tables, e)
            if layout == "two_level":
                ent.append(negf.negf_export_tables(ctx, tables, e, "alias_level1")
                           .reshape(info["rows"], L + 2))
                l2.append(negf.negf_export_tables(ctx, tables, e, "alias").view(np.uint32)
                          .reshape(info["rows"], L, negf.level2_words(W)))
            else:
                ent.append(negf.negf_export_tables(ctx, tables, e, "alias")
                           .reshape(info["rows"], info["K"]))
            ment.append(negf.negf_export_tables(ctx, tables, e, "mode_alias").reshape(2, W))
            c.append(np.asarray(info["c"]))
        energy = (tr["interval"][pick].astype(np.int64),
                  tr["a"][pick].view(np.uint32).astype(np.uint64))
        lead, steps, _, _ = thermal.walk(ent, ment, c, W * L, W, 0, 0, 77,
                                         (5 + pick).astype(np.uint64), w.energy, MU, KT, 1 << 20,
                                         energy=energy,
                                         level2=(l2, L) if layout == "two_level" else None)
        assert np.array_equal(lead, tr["lead"][pick])
        assert np.array_equal(steps, tr["steps"][pick].astype(np.uint32))
        for q in (0, 1):
            assert res["absorbed"][q] == np.count_nonzero(tr["lead"] == q)
    finally:
        negf.negf_tables_free(tables)
