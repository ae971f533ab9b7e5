"""Handles of several threads at once, each with sizes of its own: one thread's
launch must not depend on another's shared-memory size."""
import threading

import numpy as np
import pytest
import torch

from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


def _run(bodies, rounds):
    errors = []

    def loop(make):
        try:
            body = make()
            for _ in range(rounds):
                body()
        except Exception as e:   # noqa: BLE001 (reported below)
            errors.append(repr(e))

    ts = [threading.Thread(target=loop, args=(b,)) for b in bodies]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors


def _error_pass(n, k):
    def make():
        from paper_1905_13257_gb300 import IdSketch
        st = torch.cuda.Stream()
        A = gaussian_matrix(200, n, seed=n, dtype=torch.float64, device="cuda")
        sk = IdSketch(200, n, k, k, dtype=torch.float64, want_Y=False, stream=st)
        J, P = torch.arange(k), torch.zeros((k, n), dtype=torch.float64)
        torch.cuda.synchronize()
        return lambda: sk.reconstruct_error(A, J, P)
    return make


def _coarse(mc, n, k):
    def make():
        from paper_1905_13257_gb300 import IdSketch
        st = torch.cuda.Stream()
        A = gaussian_matrix(mc, n, seed=n, dtype=torch.float64, device="cuda")
        sk = IdSketch(mc, n, k, k, dtype=torch.float64, want_Y=False, grid=(1, 1, mc), ncomp=1,
                      coarse_stride=(1, 1, 1), want_coarse=True, stream=st)
        torch.cuda.synchronize()
        sk.stream_columns(A)
        sk.set_mesh(np.zeros(1), np.zeros(1), np.arange(mc) * 1.0)
        J = torch.arange(k, dtype=torch.int32)

        def body():
            assert sk.coarse_factor()[2] == k
            sk.single_pass_lift(J)
        return body
    return make


def test_error_passes_of_several_threads():
    _run([_error_pass(n, k) for n, k in ((20, 2), (100, 60), (60, 30), (150, 64))], 200)


def test_coarse_qrs_and_lifts_of_several_threads():
    _run([_coarse(mc, n, k) for mc, n, k in ((60, 20, 1), (300, 70, 40), (500, 30, 12))], 60)
