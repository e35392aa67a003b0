"""The row-group layout's orders, pieces and rules against the FP64 oracle.

The layout looks for the voxel grid's strides in the matrix and groups rows that
are neighbours along the beam, in 2 x 2 x 2 cubes, by their columns, or as they
come; groups whose union spans several packets are summed piece by piece; rows
of more than 4096 entries get the layout for the forward calls alone.  Every
route is held to the bounds of the other row-group tests: forward rows within
1e-5 relative (all terms are >= 0), g componentwise within 1e-5 (|A|^T |r|)_j, f
within 1e-12 of the oracle's f of the GPU's own dose, FP64-vector doses within
2^-40 of sum |a x|.
"""
from dataclasses import replace

import numpy as np
import pytest
import torch

import dosegen
import oracle
import paper_2103_09683_gb300 as dose
from gpu_helpers import OFMT, adj_check, fwd_check, make

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    dose.build()
    dose.load()


def _to(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _shuffled(csr, seed):
    """The same rows in random order: no strides to find."""
    order = np.random.default_rng(seed).permutation(csr.nrows)
    rp = csr.row_ptr.astype(np.int64)
    lens = np.diff(rp)[order]
    out = np.zeros(csr.nrows + 1, dtype=np.int64)
    np.cumsum(lens, out=out[1:])
    take = np.repeat(rp[:-1][order] - out[:-1], lens) + np.arange(csr.nnz)
    return dosegen.CSR(csr.nrows, csr.ncols, out.astype(np.uint32), csr.col[take], csr.val[take])


def _cases():
    """One matrix per route: along the beam (long grid, several hundred entries a
    row, so unions of more than a packet), cubes (two crossing beams), columns
    (shuffled rows), a single plane, one voxel line, and rows that fit no grid."""
    along = dosegen.generate(replace(dosegen.CLINICAL, grid=(41, 37, 48), lattice=(26, 23), spacing=(0.8, 0.8)))
    flat = dosegen.generate(replace(dosegen.TINY, grid=(61, 53, 1)))
    line = dosegen.generate(replace(dosegen.TINY, grid=(97, 1, 1), lattice=(25, 3)))
    return {"along": along, "shuffled": _shuffled(along, 3), "flat": flat, "line": line,
            "random": dosegen.random_csr(777, 301, seed=9, density=0.3, empty_frac=0.4)}


@pytest.mark.parametrize("fmt", ["u16", "fp8", "f32"])
@pytest.mark.parametrize("name", ["along", "shuffled", "flat", "line", "random"])
def test_orders_every_call(name, fmt):
    """All calls of the layout on each row order; doses written at an odd word
    offset (rows without entries then start off the 16-byte grid) leave their
    surroundings alone."""
    csr = _cases()[name]
    A, enc = make(csr, fmt)
    assert A.info()["spmv_layout"] == 2
    rng = np.random.default_rng(1)
    x = rng.uniform(0, 1, csr.ncols).astype(np.float32)
    ref = oracle.spmv(csr.nrows, enc.row_ptr, enc.col, enc.decoded, x)
    for shift in (0, 1, 3):
        buf = torch.full((csr.nrows + 8,), -3.0, dtype=torch.float32, device="cuda")
        A.spmv(_to(x), buf[shift:shift + csr.nrows])
        fwd_check(buf[shift:shift + csr.nrows].cpu().numpy(), ref)
        assert torch.all(buf[:shift] == -3.0) and torch.all(buf[shift + csr.nrows:] == -3.0)
    x64 = rng.uniform(0, 1, csr.ncols)
    d64 = A.spmv_f64(_to(x64)).cpu().numpy()
    mass = oracle.spmv(csr.nrows, enc.row_ptr, enc.col, np.abs(enc.decoded), x64)
    assert np.all(np.abs(d64 - oracle.spmv(csr.nrows, enc.row_ptr, enc.col, enc.decoded, x64)) <= 2.0 ** -40 * mass)
    r = rng.normal(size=csr.nrows).astype(np.float32)
    adj_check(A.adjoint(_to(r)).cpu().numpy(), oracle.spmv_t(csr.nrows, csr.ncols, enc.row_ptr, enc.col, enc.decoded, r),
              oracle.abs_spmv_t(csr.nrows, csr.ncols, enc.row_ptr, enc.col, enc.decoded, r))
    p = np.where(rng.uniform(size=csr.nrows) < 0.3, 2.0, 0.0).astype(np.float32)
    w = rng.uniform(0.5, 2.0, csr.nrows).astype(np.float32)
    f, g, d = A.fwd_adj_quadratic(_to(x), _to(p), _to(w), want_d=True)
    fwd_check(d.cpu().numpy(), ref)
    f_own, r_own = oracle.objective(d.cpu().numpy().astype(np.float64), p, w)
    assert abs(float(f.item()) - f_own) <= 1e-12 * max(f_own, 1e-300)
    adj_check(g.cpu().numpy(), oracle.spmv_t(csr.nrows, csr.ncols, enc.row_ptr, enc.col, enc.decoded, r_own),
              oracle.abs_spmv_t(csr.nrows, csr.ncols, enc.row_ptr, enc.col, enc.decoded, r_own))
    A.device_status()


def test_fast_order_of_the_fused_pass():
    """A beam of more than 200,000 rows with entries, whose fused pass takes the
    groups along the beam too: d, f and g against the oracle, and the rows'
    non-finite weights reach f from rows without entries."""
    csr = dosegen.generate(replace(dosegen.CLINICAL, grid=(96, 92, 73), lattice=(52, 50), sigma=2.0))
    assert np.count_nonzero(csr.row_lengths()) > 200000
    A, enc = make(csr, "u16")
    rng = np.random.default_rng(2)
    x = rng.uniform(0, 1, csr.ncols).astype(np.float32)
    p = np.where(rng.uniform(size=csr.nrows) < 0.1, 2.0, 0.0).astype(np.float32)
    w = rng.uniform(0.5, 2.0, csr.nrows).astype(np.float32)
    f, g, d = A.fwd_adj_quadratic(_to(x), _to(p), _to(w), want_d=True)
    fwd_check(d.cpu().numpy(), oracle.spmv(csr.nrows, enc.row_ptr, enc.col, enc.decoded, x))
    f_own, r_own = oracle.objective(d.cpu().numpy().astype(np.float64), p, w)
    assert abs(float(f.item()) - f_own) <= 1e-12 * f_own
    adj_check(g.cpu().numpy(), oracle.spmv_t(csr.nrows, csr.ncols, enc.row_ptr, enc.col, enc.decoded, r_own),
              oracle.abs_spmv_t(csr.nrows, csr.ncols, enc.row_ptr, enc.col, enc.decoded, r_own))
    empty = np.flatnonzero(csr.row_lengths() == 0)
    for bad in (np.inf, np.nan):
        w2 = w.copy()
        w2[empty[len(empty) // 2]] = bad
        p2 = p.copy()
        p2[empty[len(empty) // 2]] = 0.0
        f2, _ = A.fwd_adj_quadratic(_to(x), _to(p2), _to(w2))
        assert np.isnan(float(f2.item()))  # 0 * inf, 0 * nan
    A.device_status()


@pytest.mark.parametrize("fmt", ["u16", "f16"])
def test_long_rows_forward_only(fmt):
    """Neighbouring rows of 4000-5200 of 6000 columns: the layout serves dose_spmv,
    dose_spmv_f64 and the batch; asked for explicitly it is refused as before, and
    the adjoint stays on CSR."""
    rng = np.random.default_rng(4)
    base = rng.permutation(6000)
    rows = [np.sort(base[:int(n)]) for n in rng.integers(4000, 5200, 41)]
    rows[5] = rows[17] = np.zeros(0, dtype=np.int64)
    rp = np.concatenate([[0], np.cumsum([len(c) for c in rows])]).astype(np.uint32)
    col = np.concatenate(rows).astype(np.uint32)
    csr = dosegen.CSR(len(rows), 6000, rp, col, rng.uniform(0.1, 1.0, col.size))
    A, enc = make(csr, fmt)
    info = A.info()
    assert info["max_row_len"] > 4096 and info["spmv_layout"] == 2 and info["adj_layout_adjoint"] == 1
    x = rng.uniform(0, 1, 6000).astype(np.float32)
    # a lane of the warp adds at most ceil(nu / 32) terms of a row, then five levels
    fwd_check(A.spmv(_to(x)).cpu().numpy(), oracle.spmv(csr.nrows, rp, col, enc.decoded, x), rtol=(188 + 6) * 2.0 ** -24)
    x64 = rng.uniform(0, 1, 6000)
    ref = oracle.spmv(csr.nrows, rp, col, enc.decoded, x64)
    assert np.all(np.abs(A.spmv_f64(_to(x64)).cpu().numpy() - ref) <= 2.0 ** -40 * ref)
    for tuning in (dict(adj_layout=2), dict(fwd_layout=2)):
        with pytest.raises(dose.DoseError) as ei:
            make(csr, fmt, tuning=tuning)
        assert ei.value.status == 4
    r = rng.normal(size=csr.nrows).astype(np.float32)
    adj_check(A.adjoint(_to(r)).cpu().numpy(), oracle.spmv_t(csr.nrows, 6000, rp, col, enc.decoded, r),
              oracle.abs_spmv_t(csr.nrows, 6000, rp, col, enc.decoded, r))
    A.device_status()


def test_batch_of_both_group_heights():
    """One batch of matrices with eight-row and four-row groups: two launches, and
    every D within the bound."""
    mats = [_cases()["along"], dosegen.random_csr(900, 301, seed=10, density=0.1, empty_frac=0.5), _cases()["flat"]]
    hs, encs, Xs = [], [], []
    for i, m in enumerate(mats):
        A, enc = make(m, "u16")
        hs.append(A)
        encs.append(enc)
        Xs.append(_to(dosegen.spot_weights(m.ncols, 70 + i, nvec=7).reshape(m.ncols, 7)))
    layout, launches = dose.spmv_batched_plan(hs, 7)
    assert layout == 2 and launches in (1, 2)
    for m, enc, X, D in zip(mats, encs, Xs, dose.spmv_batched(hs, Xs)):
        ref = oracle.spmm(m.nrows, enc.row_ptr, enc.col, enc.decoded, X.cpu().numpy().astype(np.float64))
        fwd_check(D.cpu().numpy().reshape(-1), ref.reshape(-1))


def test_robust_set_with_a_matrix_twice():
    """Overlapped scenario passes against the sequence of single passes: a set of
    distinct matrices gives each scenario's f and the mean gradient of the single
    calls, and a set that lists one matrix twice (never overlapped) agrees."""
    beams = [replace(dosegen.TINY, shift=s) for s in ((0.0, 0.0), (-3.0, 0.0), (3.0, 3.0))]
    As = [make(dosegen.generate(b), "u16")[0] for b in beams]
    p, w = (_to(a) for a in dosegen.ellipsoid_target(dosegen.TINY))
    x = _to(dosegen.spot_weights(As[0].ncols, 5))
    single = [A.fwd_adj_quadratic(x, p, w) for A in As]
    for mats in (As, [As[0], As[1], As[0]]):
        fs = torch.empty(3, dtype=torch.float64, device="cuda")
        f, g, _ = dose.ScenarioSet(mats).robust_quadratic(x, p, w, mode="expected", f_scen=fs)
        idx = [As.index(A) for A in mats]
        for k, i in enumerate(idx):
            assert fs[k].item() == single[i][0].item()
        mean = torch.stack([single[i][1].double() for i in idx]).mean(0)
        assert torch.all((g.double() - mean).abs() <= 2e-7 * mean.abs().max())


def test_compensated_rows_at_lane_edges():
    """Compensated sums with rows of 1 to 300 entries side by side (some warps hold
    rows on both sides of 128) and every start offset within a 16-byte piece."""
    lens = np.concatenate([np.arange(1, 12), [127, 128, 129, 130, 131, 255, 256, 257, 300], [0, 3, 129, 2, 140]])
    csr = dosegen.random_csr(len(lens), 400, seed=21, lengths=lens)
    for fmt in ("f32", "u16", "fp8"):
        for index16 in (False, True):
            A, enc = make(csr, fmt, compensated=True, index16=index16)
            x = np.random.default_rng(6).uniform(0, 1, 400).astype(np.float32)
            fwd_check(A.spmv(_to(x)).cpu().numpy(), oracle.spmv(csr.nrows, enc.row_ptr, enc.col, enc.decoded, x))
