"""Slices wider than 16 sites in FP32 against the oracle: the sweeps' and diagonal blocks' panel
inversions (four pivots a panel: widths of every remainder, both column halves, the ends of the
range), slices that take the pivoted fallback between dephased ones, multi-orbital slice blocks
and sweeps of one slice.  Bar: weights elementwise within 1e-5 of the row sum (the FP32 table
bar), row sums and Tr[Gamma A] to 1e-5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import pipeline  # noqa: E402
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


def _undephased(w):
    w.eta = w.eta.copy()
    w.eta[1, ::3] = 0.0
    w.eta[3, :] = 0.0
    return w


CASES = {f"W{W}_L{L}": (lambda W=W, L=L: inputs.small_wire(500 + W, W, L, n_energy=2, eta=0.05,
                                                          disorder=0.7, e_lo=-1.7, e_hi=1.3))
         for W, L in ((17, 2), (18, 5), (19, 4), (32, 3), (33, 2), (34, 5), (35, 3), (36, 1),
                      (45, 6), (61, 3), (62, 2), (63, 4), (64, 5))}
CASES.update({f"undephased_W{W}": (lambda W=W: _undephased(
    inputs.small_wire(600 + W, W, 6, n_energy=1, eta=0.08, disorder=0.8, e_lo=0.3, e_hi=0.3)))
    for W in (21, 32, 38, 64)})
CASES["orbitals_W36"] = lambda: inputs.sp3_wire(611, 9, 4, n_energy=2, eta=0.08)
CASES["orbitals_W20"] = lambda: _undephased(inputs.sp3_wire(612, 5, 5, n_energy=1, eta=0.08))
CASES["wide_band_W40"] = lambda: inputs.small_wire(613, 40, 4, n_energy=1, eta=0.05,
                                                  lead_model=1, gamma_lead=0.7)


@pytest.mark.parametrize("name", list(CASES))
def test_wide_slices_match_oracle(ctx, name):
    w = CASES[name]()
    tables = negf.negf_build_tables(ctx, [w], precision="fp32", keep_weights=True)
    try:
        for task, E in enumerate(w.energy):
            ref = pipeline.task_reference(w.onsite, w.eta, w.t, E, w.lead_model, w.gamma_lead,
                                          with_alias=False, slice_h=w.slice_h)
            w_ref = ref["tab"]["w"]
            rs_ref = w_ref.sum(1)
            got = negf.negf_export_tables(ctx, tables, task, "weights").reshape(w_ref.shape)
            assert np.all(np.abs(got - w_ref) <= 1e-5 * rs_ref[:, None] + 1e-30), task
            rs = negf.negf_export_tables(ctx, tables, task, "rowsum")
            assert np.allclose(rs, rs_ref, rtol=1e-5), task
            assert np.allclose(negf.negf_get_task_info(ctx, tables, task)["c"], ref["tab"]["c"],
                               rtol=1e-5), task
    finally:
        negf.negf_tables_free(tables)
