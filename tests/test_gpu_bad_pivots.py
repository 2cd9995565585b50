"""Complex64 slices wider than 16 sites with a pivot that has no finite reciprocal (an onsite energy
beyond the FP32 range), in the first, a middle and the last slice: every thread of a sweep has to
see that inversion's flag, and no later one's, so that the sweep ends as a whole; the call reports
a singular slice block, and the next build on the context gives the tables it gave before."""
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


def _rows(ctx, wire):
    tables = negf.negf_build_tables(ctx, [wire], precision="fp32", keep_weights=True)
    try:
        return [negf.negf_export_tables(ctx, tables, k, "weights") for k in range(len(wire.energy))]
    finally:
        negf.negf_tables_free(tables)


@pytest.mark.parametrize("k_bad", [0, 3, 6])
@pytest.mark.parametrize("W", [17, 32, 33, 64])
def test_pivot_without_finite_reciprocal(ctx, W, k_bad):
    wire = inputs.small_wire(800 + W, W, 7, n_energy=2, eta=0.05)
    before = _rows(ctx, wire)
    bad = inputs.small_wire(800 + W, W, 7, n_energy=2, eta=0.05)
    bad.onsite = bad.onsite.copy()
    bad.onsite[k_bad, W // 2] = 1e39
    tables = negf.negf_build_tables(ctx, [bad], precision="fp32")
    try:
        with pytest.raises(negf.NegfError, match="singular slice block") as e:
            negf.negf_get_task_info(ctx, tables, 0)
        assert e.value.status == negf.NEGF_E_NUMERIC
    finally:
        negf.negf_tables_free(tables)
    for a, b in zip(before, _rows(ctx, wire)):
        assert np.array_equal(a, b)
