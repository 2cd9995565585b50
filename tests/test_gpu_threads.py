"""Threads, each with its own context and stream, building batches whose alias rows fall into
several classes (the row kernel is launched with another amount of shared memory for each): no
launch is refused for a limit that another thread has set, and every table is what it is alone.
A plan whose waves launch that kernel with different amounts gives the same counts before and
after builds that need little shared memory."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1805_10164_gb300 import inputs, negf  # noqa: E402


def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_10164_gb300 import build
    build.build()


def _wire(W, L, n_energy=1):
    return inputs.small_wire(720 + W + L, W, L, n_energy=n_energy, eta=0.06, disorder=0.8,
                             e_lo=0.2, e_hi=0.5)


BATCHES = [([(1, 30), (2, 549)], "fp32"), ([(1, 20)], "fp32"), ([(1, 30), (2, 300)], "fp64"),
           ([(3, 9)], "fp64")]


def _rows(ctx, sizes, precision):
    tables = negf.negf_build_tables(ctx, [_wire(W, L) for W, L in sizes], precision=precision,
                                    layout="one_level")
    try:
        return [negf.negf_export_tables(ctx, tables, k, "alias") for k in range(len(sizes))]
    finally:
        negf.negf_tables_free(tables)


def test_threads_build_side_by_side():
    _need_gpu()
    ctx = negf.negf_create(0)
    want = [_rows(ctx, *b) for b in BATCHES]
    negf.negf_destroy(ctx)
    errors = []

    def work(first):
        try:
            torch.cuda.set_device(0)
            c = negf.negf_create(0, torch.cuda.Stream())
            for i in range(300):
                k = (i + first) % len(BATCHES)
                for a, b in zip(want[k], _rows(c, *BATCHES[k])):
                    assert np.array_equal(a, b), k
            negf.negf_destroy(c)
        except Exception as e:          # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(f,)) for f in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


def test_plan_after_builds_of_little_shared_memory():
    _need_gpu()
    ctx = negf.negf_create(0)
    wires = [_wire(2, 549, 2), _wire(1, 30, 2)]
    plan = negf.negf_plan_create(ctx, wires, 0, 5000, 0.6, -0.4, 0.3, tasks_per_wave=2,
                                 layout="one_level")
    try:
        negf.negf_plan_launch(ctx, plan, 5)
        first = negf.negf_plan_result(ctx, plan)["counts"]
        _rows(ctx, [(1, 20)], "fp32")
        negf.negf_plan_launch(ctx, plan, 5)
        assert np.array_equal(first, negf.negf_plan_result(ctx, plan)["counts"])
    finally:
        negf.negf_plan_destroy(plan)
        negf.negf_destroy(ctx)
