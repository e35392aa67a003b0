"""Calls queued back to back, each of which reads what the one before it has just
written: the row-group kernels start while their predecessor still runs, so the
results must be those of the same calls with a synchronisation after each, bit for
bit.  x lies off the 32-byte grid, so that blocks of two SMs write one sector of it."""
from dataclasses import replace

import numpy as np
import pytest
import torch

import dosegen
import paper_2103_09683_gb300 as dose
from gpu_helpers import make

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    dose.build()
    dose.load()


def _to(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _at(a, shift):
    """A copy of `a` that starts `shift` elements into its allocation."""
    t = _to(a)
    buf = torch.zeros(t.numel() + shift, dtype=t.dtype, device="cuda")
    buf[shift:] = t
    return buf[shift:]


@pytest.mark.parametrize("shift", [0, 1, 5])
@pytest.mark.parametrize("fmt", ["u16", "fp8"])
def test_projected_gradient_steps(fmt, shift):
    csr = dosegen.generate(dosegen.TINY)
    A, _ = make(csr, fmt)
    p, w = (_to(a) for a in dosegen.ellipsoid_target(dosegen.TINY))
    runs = []
    for sync in (True, False):
        x = _at(dosegen.spot_weights(csr.ncols, 9), shift)
        f = torch.zeros(150, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        for k in range(150):
            A.pg_step(x, p, w, 1e-6, f=f[k:k + 1])
            if sync:
                torch.cuda.synchronize()
        runs.append((f, x.clone()))
    assert float(runs[0][0][-1]) != float(runs[0][0][0])
    for a, b in zip(*runs):
        assert torch.equal(a, b)
    A.device_status()


@pytest.mark.parametrize("fmt", ["u16", "bf16", "f32"])
def test_forward_and_adjoint_in_turn(fmt):
    """d = A x into the adjoint's r, g = A^T r into the next x (a power iteration on a
    matrix of norm at most 1), and the batched form of the same x."""
    csr = dosegen.generate(replace(dosegen.TINY, grid=(41, 37, 24)))
    cols = np.bincount(csr.col, weights=csr.val, minlength=csr.ncols).max()
    rows = np.bincount(np.repeat(np.arange(csr.nrows), csr.row_lengths()), weights=csr.val).max()
    csr = dosegen.CSR(csr.nrows, csr.ncols, csr.row_ptr, csr.col, csr.val / np.sqrt(rows * cols))
    A, _ = make(csr, fmt)
    runs = []
    for sync in (True, False):
        x = _at(dosegen.spot_weights(csr.ncols, 11), 3)
        d = torch.empty(csr.nrows, dtype=torch.float32, device="cuda")
        D = [torch.empty((csr.nrows, 1), dtype=torch.float32, device="cuda") for _ in range(60)]
        torch.cuda.synchronize()
        for k in range(60):
            A.spmv(x, d)
            if sync:
                torch.cuda.synchronize()
            A.adjoint(d, x)
            if sync:
                torch.cuda.synchronize()
            dose.spmv_batched([A], [x.view(-1, 1)], [D[k]])
            if sync:
                torch.cuda.synchronize()
        runs.append([x.clone(), d] + D)
    assert float(runs[0][0].abs().max()) > 0
    for a, b in zip(*runs):
        assert torch.equal(a, b)
    A.device_status()
