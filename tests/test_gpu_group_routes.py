"""Which row order and group height the row-group layout took, and the eight-row
fused pass on each of them: dose_info says both, so that every case here is known to
run on the route it names.  Bounds as in the other row-group tests: doses within
1e-5 relative (all terms are >= 0), g componentwise within 1e-5 (|A|^T |r|)_j, f
within 1e-12 of the oracle's f of the GPU's own dose."""
from dataclasses import replace

import numpy as np
import pytest
import torch

import dosegen
import oracle
import paper_2103_09683_gb300 as dose
from gpu_helpers import OFMT, adj_check, fwd_check, make

pytestmark = pytest.mark.gpu

AS_STORED, PLANES, CUBES, COLUMNS = range(4)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    dose.build()
    dose.load()


def _to(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _plan(grid, lattice):
    """The three beams of a plan (along z, x and y), and their merged matrix."""
    beams = [dosegen.generate_along(b, a) for b, a in dosegen.robust_plan(grid, lattice)[0]]
    lens = sum(b.row_lengths().astype(np.int64) for b in beams)
    rp = np.zeros(beams[0].nrows + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    col, val = np.empty(rp[-1], dtype=np.uint32), np.empty(rp[-1])
    at, base = rp[:-1].copy(), 0
    for b in beams:
        n = b.row_lengths().astype(np.int64)
        pos = np.repeat(at - b.row_ptr[:-1].astype(np.int64), n) + np.arange(b.nnz)
        col[pos], val[pos] = b.col + base, b.val
        at, base = at + n, base + b.ncols
    return beams, dosegen.CSR(beams[0].nrows, base, rp.astype(np.uint32), col, val)


def _check(A, csr, enc):
    rng = np.random.default_rng(2)
    x = rng.uniform(0, 1, csr.ncols).astype(np.float32)
    p = np.where(rng.uniform(size=csr.nrows) < 0.1, 2.0, 0.0).astype(np.float32)
    w = rng.uniform(0.5, 2.0, csr.nrows).astype(np.float32)
    ref = oracle.spmv(csr.nrows, enc.row_ptr, enc.col, enc.decoded, x)
    fwd_check(A.spmv(_to(x)).cpu().numpy(), ref)
    f, g, d = A.fwd_adj_quadratic(_to(x), _to(p), _to(w), want_d=True)
    fwd_check(d.cpu().numpy(), ref)
    f_own, r_own = oracle.objective(d.cpu().numpy().astype(np.float64), p, w)
    assert abs(float(f.item()) - f_own) <= 1e-12 * f_own
    g_ref = oracle.spmv_t(csr.nrows, csr.ncols, enc.row_ptr, enc.col, enc.decoded, r_own)
    g_abs = oracle.abs_spmv_t(csr.nrows, csr.ncols, enc.row_ptr, enc.col, enc.decoded, r_own)
    adj_check(g.cpu().numpy(), g_ref, g_abs)
    adj_check(A.adjoint(_to(r_own.astype(np.float32))).cpu().numpy(), g_ref, g_abs)
    A.device_status()


def _route(name):
    if name == "planes":  # one beam, deep grid
        return dosegen.generate(replace(dosegen.CLINICAL, grid=(64, 60, 73), lattice=(32, 30), sigma=2.0))
    if name == "cubes":  # crossing beams
        return _plan((40, 44, 36), (12, 10))[1]
    if name == "columns":  # no strides, rows that share columns are not neighbours
        return dosegen.random_csr(777, 301, seed=9, density=0.3, empty_frac=0.4)
    return dosegen.generate(replace(dosegen.TINY, grid=(61, 53, 1)))  # one plane: as stored


@pytest.mark.parametrize("name,order,rows", [("planes", PLANES, 8), ("cubes", CUBES, 8), ("columns", COLUMNS, 4),
                                             ("stored", AS_STORED, 8)])
def test_route_of_each_order(name, order, rows):
    csr = _route(name)
    A, enc = make(csr, "u16")
    info = A.info()
    assert (info["rg_order"], info["rg_rows"]) == (order, rows)
    _check(A, csr, enc)
    assert make(csr, "f32")[0].info()["rg_rows"] == 4


@pytest.mark.parametrize("nvec", [1, 7, 16])
def test_batch_of_both_heights_takes_two_launches(nvec):
    mats = [_route("cubes"), _route("columns"), _route("stored")]
    hs, encs = zip(*(make(m, "u16") for m in mats))
    assert {A.info()["rg_rows"] for A in hs} == {4, 8}
    assert dose.spmv_batched_plan(list(hs), nvec) == (2, 2)
    Xs = [_to(dosegen.spot_weights(m.ncols, 70 + i, nvec=nvec).reshape(m.ncols, nvec)) for i, m in enumerate(mats)]
    for m, enc, X, D in zip(mats, encs, Xs, dose.spmv_batched(list(hs), Xs)):
        ref = oracle.spmm(m.nrows, enc.row_ptr, enc.col, enc.decoded, X.cpu().numpy().astype(np.float64))
        fwd_check(D.cpu().numpy().reshape(-1), ref.reshape(-1))


@pytest.fixture(scope="module")
def large_beams():
    """More than 200,000 rows with entries: the fused pass runs on the layout's own
    groups.  Rows of up to 71 entries, and of up to 419 (groups of several packets)."""
    short = dosegen.generate(replace(dosegen.CLINICAL, grid=(96, 92, 73), lattice=(52, 50), sigma=2.0))
    long = dosegen.generate(replace(dosegen.CLINICAL, grid=(90, 86, 60), lattice=(64, 60), spacing=(1.0, 1.0)))
    assert min(np.count_nonzero(c.row_lengths()) for c in (short, long)) > 200000 and long.row_lengths().max() > 320
    return short, long


@pytest.mark.parametrize("fmt", ["u16", "bf16", "f16", "fp8", "f32"])
@pytest.mark.parametrize("which", [0, 1])
def test_fused_pass_of_large_beams(large_beams, which, fmt):
    csr = large_beams[which]
    A, enc = make(csr, fmt)
    assert A.info()["rg_rows"] == (4 if fmt == "f32" else 8) and A.info()["adj_layout_fused"] == 2
    _check(A, csr, enc)


@pytest.mark.parametrize("fmt", ["f16", "bf16"])
def test_fused_pass_of_a_large_plan(fmt):
    """A merged plan of more than 400,000 rows with entries."""
    beams, csr = _plan((128, 128, 96), (30, 20))
    assert np.count_nonzero(csr.row_lengths()) > 400000
    encs = [oracle.encode(b, OFMT[fmt]) for b in beams]
    A = dose.DoseMatrix.from_multibeam([(e.row_ptr, e.col, e.ncols, e.values, None) for e in encs], fmt=fmt)
    assert (A.info()["rg_order"], A.info()["rg_rows"]) == (CUBES, 8)
    _check(A, csr, oracle.encode(csr, OFMT[fmt]))


@pytest.mark.parametrize("fmt", ["u16", "fp8", "f32"])
def test_fused_pass_of_medium_beams(fmt):
    """Between 100,000 and 200,000 rows with entries: the stored-row groups on the other
    layout's deal (FP8: on their own)."""
    csr = _route("planes")
    assert 100000 < np.count_nonzero(csr.row_lengths()) < 200000
    A, enc = make(csr, fmt)
    _check(A, csr, enc)


@pytest.mark.parametrize("fmt", ["bf16", "f32"])
def test_fused_pass_of_a_medium_plan(fmt):
    """100,000 to 400,000 rows with entries, unions of several packets; a second call
    gives the same bits."""
    beams, csr = _plan((72, 70, 50), (18, 12))
    assert 100000 < np.count_nonzero(csr.row_lengths()) < 400000 and csr.row_lengths().max() > 320
    encs = [oracle.encode(b, OFMT[fmt]) for b in beams]
    A = dose.DoseMatrix.from_multibeam([(e.row_ptr, e.col, e.ncols, e.values, None) for e in encs], fmt=fmt)
    _check(A, csr, oracle.encode(csr, OFMT[fmt]))
    x, p, w = (_to(np.random.default_rng(k).uniform(0, 1, n).astype(np.float32))
               for k, n in ((1, csr.ncols), (2, csr.nrows), (3, csr.nrows)))
    for a, b in zip(A.fwd_adj_quadratic(x, p, w, want_d=True), A.fwd_adj_quadratic(x, p, w, want_d=True)):
        assert torch.equal(a, b)
