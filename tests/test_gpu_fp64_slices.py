"""FP64 tables over the widths at which the sweeps change their rows per thread and over wires of
one to a few slices (chains towards slice 0, each block and its transpose, the lead weights from
the injection columns), against the oracle.  Bar: weights elementwise within 1e-10 relative and
1e-13 of the row sum (the FP64 table bar), row sums and Tr[Gamma A] to 1e-10."""
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
    return w


CASES = {f"W{W}_L{L}": (lambda W=W, L=L: inputs.small_wire(800 + W, W, L, n_energy=2, eta=0.06,
                                                          disorder=0.7, e_lo=-1.7, e_hi=1.3))
         for W, L in ((1, 1), (1, 2), (2, 7), (3, 4), (4, 1), (11, 6), (12, 3), (16, 5), (17, 2),
                      (22, 4), (23, 3), (32, 3), (33, 2), (42, 3), (43, 2), (64, 3))}
CASES["undephased_W16"] = lambda: _undephased(inputs.small_wire(851, 16, 5, n_energy=1, eta=0.08))
CASES["orbitals_W20"] = lambda: inputs.sp3_wire(852, 5, 4, n_energy=2, eta=0.08)
CASES["wide_band_W9"] = lambda: inputs.small_wire(853, 9, 6, n_energy=1, eta=0.05, lead_model=1,
                                                  gamma_lead=0.7)


@pytest.mark.parametrize("name", list(CASES))
def test_fp64_slices_match_oracle(ctx, name):
    w = CASES[name]()
    tables = negf.negf_build_tables(ctx, [w], precision="fp64", keep_weights=True)
    try:
        for task, E in enumerate(w.energy):
            ref = pipeline.task_reference(w.onsite, w.eta, w.t, E, w.lead_model, w.gamma_lead,
                                          with_alias=False, slice_h=w.slice_h)
            w_ref = ref["tab"]["w"]
            rs_ref = w_ref.sum(1)
            got = negf.negf_export_tables(ctx, tables, task, "weights").reshape(w_ref.shape)
            assert np.all(np.abs(got - w_ref) <= 1e-10 * w_ref + 1e-13 * rs_ref[:, None]), task
            rs = negf.negf_export_tables(ctx, tables, task, "rowsum")
            assert np.allclose(rs, rs_ref, rtol=1e-10, atol=1e-300), task
            info = negf.negf_get_task_info(ctx, tables, task)
            assert np.allclose(info["c"], ref["tab"]["c"], rtol=1e-10), task
    finally:
        negf.negf_tables_free(tables)
