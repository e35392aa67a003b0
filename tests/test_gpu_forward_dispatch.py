"""Where the forward calls take row groups by default and where CSR: few warps beside a
wide list of columns, and many stored zeros for the FP64-vector form.  Each handle is
compared with one that was told which layout to take, and with the FP64 oracle."""
import numpy as np
import pytest
import torch

import dosegen
import oracle
import paper_2103_09683_gb300 as dose
from gpu_helpers import fwd_check, make

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    dose.build()
    dose.load()


def _to(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _scattered(nrows, ncols, per_row, seed, alike=1):
    """per_row entries a row, one in each of per_row equal parts of the columns;
    `alike` neighbouring rows share them."""
    rng = np.random.default_rng(seed)
    lo = np.arange(per_row + 1, dtype=np.int64) * ncols // per_row
    col = lo[:-1] + (rng.random((nrows // alike, per_row)) * (lo[1:] - lo[:-1])).astype(np.int64)
    col = np.repeat(col, alike, axis=0).reshape(-1).astype(np.uint32)
    rp = (per_row * np.arange(nrows + 1, dtype=np.int64)).astype(np.uint32)
    return dosegen.CSR(nrows, ncols, rp, col, rng.uniform(0.1, 1.0, col.size))


def test_one_warp_beside_x_is_left_to_csr():
    """About 54,500 of 65,000 columns a CTA: one warp fits.  CSR by default; row groups
    where they are asked for, with the same dose within the bound."""
    csr = _scattered(60000, 65000, 300, 1)
    x = np.random.default_rng(2).uniform(0, 1, csr.ncols).astype(np.float32)
    A, enc = make(csr, "u16")
    B, _ = make(csr, "u16", tuning=dict(fwd_layout=2))
    assert A.info()["rg_window"] > 52000
    assert A.info()["spmv_layout"] == 1 and B.info()["spmv_layout"] == 2
    ref = oracle.spmv(csr.nrows, enc.row_ptr, enc.col, enc.decoded, x)
    for H in (A, B):
        fwd_check(H.spmv(_to(x)).cpu().numpy(), ref)
        H.device_status()


@pytest.mark.parametrize("ncols", [20000, 40000])
def test_wide_lists_stay_on_row_groups(ncols):
    csr = _scattered(24000, ncols, 300, 3)
    x = np.random.default_rng(4).uniform(0, 1, ncols).astype(np.float32)
    A, enc = make(csr, "u16")
    assert A.info()["spmv_layout"] == 2
    fwd_check(A.spmv(_to(x)).cpu().numpy(), oracle.spmv(csr.nrows, enc.row_ptr, enc.col, enc.decoded, x))
    A.device_status()


def _combs():
    """Rows of 1000 entries in fours; 24 neighbouring fours see 24,000 columns between
    them, so that every CTA does."""
    n = 152 * 24 * 4
    col = ((np.arange(n) // 4 % 24)[:, None] + 24 * np.arange(1000)).astype(np.uint32).reshape(-1)
    return dosegen.CSR(n, 24000, (1000 * np.arange(n + 1)).astype(np.uint32), col,
                       np.random.default_rng(7).uniform(0.1, 1.0, col.size))


@pytest.mark.parametrize("name,fmt,layout", [("alone", "f16", 1), ("alike", "f16", 2), ("combs", "f32", 1), ("small", "f16", 2)])
def test_fp64_vectors_take_the_cheaper_layout(name, fmt, layout):
    """Rows alone in their groups store four values per entry: CSR.  Eight alike store
    one: row groups, but not where three warps fit (combs).  A small matrix is left on
    row groups whatever it stores."""
    csr = (_combs() if name == "combs" else _scattered(20000, 8000, 300, 5) if name == "alone"
           else _scattered(40000, 6000, 150, 6, alike=8) if name == "alike" else _scattered(900, 3000, 200, 8))
    x = np.random.default_rng(9).uniform(0, 1, csr.ncols)
    A, enc = make(csr, fmt)
    assert A.info()["spmv_layout"] == 2
    got = A.spmv_f64(_to(x))
    told = [make(csr, fmt, tuning=dict(fwd_layout=k))[0].spmv_f64(_to(x)) for k in (1, 2)]
    assert not torch.equal(told[0], told[1])  # (they add in other orders)
    assert torch.equal(got, told[layout - 1])
    ref = oracle.spmv(csr.nrows, enc.row_ptr, enc.col, enc.decoded, x)
    assert np.all(np.abs(got.cpu().numpy() - ref) <= 2.0 ** -40 * ref)
    A.device_status()


def test_forward_layout_that_no_call_takes_is_not_kept():
    """Eight rows of 32,768 entries whose group sees 58,768 columns: it would store less
    than CSR, but its columns of x fit no CTA."""
    starts = [0, 13000, 26000] + [26000] * 5
    col = np.concatenate([np.arange(s, s + 32768) for s in starts]).astype(np.uint32)
    rp = (32768 * np.arange(9)).astype(np.uint32)
    rng = np.random.default_rng(10)
    csr = dosegen.CSR(8, 60000, rp, col, rng.uniform(0.1, 1.0, col.size))
    A, enc = make(csr, "u16")
    assert A.info()["rg_groups"] == 0 and A.info()["spmv_layout"] == 1
    x = rng.uniform(0, 1, 60000).astype(np.float32)
    # 32 lanes of four accumulators: ceil(32768 / 128) + 2 + 5 roundings of a term
    fwd_check(A.spmv(_to(x)).cpu().numpy(), oracle.spmv(8, rp, col, enc.decoded, x), rtol=(256 + 7) * 2.0 ** -24)
    A.device_status()
