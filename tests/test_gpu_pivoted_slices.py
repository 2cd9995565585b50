"""Wide complex64 slices with undephased sites (partial pivoting, the block exchanged between two
buffers a pivot: every parity of the width and of its panels) between dephased ones: tables
against the oracle (elementwise 1e-5 of the row sum, the FP32 table bar), and the block-column
adjoint, whose sweeps share the inversion, with exact tallies against the oracle's derivative
(the FP32 bars of test_gpu_gradient_rgf; the rates of undephased sites are left out: no walk
reaches such a site, so no count carries its derivative)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import test_gpu_gradient_rgf as rgf  # noqa: E402
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


def _wire(W, L, eta):
    w = inputs.small_wire(640 + W, W, L, n_energy=1, eta=eta, disorder=0.8, e_lo=0.3, e_hi=0.3)
    w.eta = w.eta.copy()
    w.eta[1, ::3] = 0.0
    w.eta[3, :] = 0.0
    w.eta[4, W // 2] = 0.0
    return w


@pytest.mark.parametrize("W", [17, 18, 24, 31, 33, 50, 63])
def test_tables(ctx, W):
    w = _wire(W, 6, 0.08)
    tables = negf.negf_build_tables(ctx, [w], precision="fp32", keep_weights=True)
    try:
        ref = pipeline.task_reference(w.onsite, w.eta, w.t, w.energy[0], with_alias=False)
        w_ref = ref["tab"]["w"]
        got = negf.negf_export_tables(ctx, tables, 0, "weights").reshape(w_ref.shape)
        assert np.all(np.abs(got - w_ref) <= 1e-5 * w_ref.sum(1)[:, None] + 1e-30)
    finally:
        negf.negf_tables_free(tables)


@pytest.mark.parametrize("W,L", [(3, 6), (7, 6), (18, 5)])
def test_adjoint(ctx, W, L):
    w = _wire(W, L, 0.2)
    tables = negf.negf_build_tables(ctx, [w], precision="fp32", keep_weights=True)
    tally = rgf._exact_tally(ctx, tables, w, 0)
    try:
        dV, dE, _ = negf.negf_current_backward_rgf(ctx, tables, tally, rgf.MU_P, rgf.MU_Q, rgf.KT,
                                                   [1.0], W * L)
        gV, gE = rgf._exact_grad(w, 0)
        scale = max(np.abs(gV).max(), np.abs(gE).max())
        live = w.eta.reshape(-1) > 0
        rgf._check(dV, gV, "fp32", scale, "dV")
        rgf._check(dE[live], gE[live], "fp32", scale, "deta")
    finally:
        negf.negf_tally_free(tally)
        negf.negf_tables_free(tables)
