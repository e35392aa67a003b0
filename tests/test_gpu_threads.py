"""Calls of one kernel from several host threads, with matrices that need different
amounts of shared memory: no call may change what another one is allowed."""
import threading

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


@pytest.mark.parametrize("fwd_layout", [0, 1])
def test_matrices_of_different_widths_side_by_side(fwd_layout):
    """The wide matrix's window of x takes twice the narrow one's shared memory.  Every
    call is accepted and gives what it gives alone."""
    handles, xs, ref = [], [], []
    for ncols in (600, 12000):
        csr = dosegen.random_csr(2000, ncols, seed=ncols, density=30 / ncols)
        A, _ = make(csr, "u16", tuning=dict(fwd_layout=fwd_layout) if fwd_layout else None)
        x = torch.from_numpy(np.random.default_rng(1).uniform(0, 1, ncols).astype(np.float32)).cuda()
        handles.append(A)
        xs.append(x)
        ref.append(A.spmv(x))
    torch.cuda.synchronize()
    wrong = []

    def work(k):
        s = torch.cuda.Stream()
        d = torch.empty_like(ref[k])
        try:
            for _ in range(3000):
                handles[k].spmv(xs[k], d, stream=s)
            s.synchronize()
            if not torch.equal(d, ref[k]):
                wrong.append("another dose")
        except Exception as e:
            wrong.append(repr(e))

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
    for A in handles:
        A.device_status()
