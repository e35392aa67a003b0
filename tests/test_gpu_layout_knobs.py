"""The row-group layout's reported knobs on rows that span several packets (more
than 320 entries): what dose_info reports can be given back to dose_set_tuning, to
a new handle and to the autotuner's cache, and a refused value changes nothing."""
import numpy as np
import pytest
import torch

import dosegen
import oracle
import paper_2103_09683_gb300 as dose
from gpu_helpers import adj_check, fwd_check, make

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    dose.build()
    dose.load()


def _to(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _long_rows():
    """330 to 1000 entries a row, a third of the rows empty."""
    rng = np.random.default_rng(12)
    lens = rng.integers(330, 1001, 400)
    lens[rng.uniform(size=400) < 0.33] = 0
    return dosegen.random_csr(400, 1200, seed=12, lengths=lens)


def _outputs(A, csr):
    rng = np.random.default_rng(3)
    x = _to(rng.uniform(0, 1, csr.ncols).astype(np.float32))
    p = _to(np.where(rng.uniform(size=csr.nrows) < 0.3, 60.0, 0.0).astype(np.float32))
    w = _to(rng.uniform(0.5, 2.0, csr.nrows).astype(np.float32))
    r = _to(rng.normal(size=csr.nrows).astype(np.float32))
    f, g, d = A.fwd_adj_quadratic(x, p, w, want_d=True)
    return [A.spmv(x), f, g, d, A.adjoint(r)]


@pytest.mark.parametrize("fmt", ["u16", "fp8", "f32"])
def test_reported_knobs_are_taken_back(fmt):
    csr = _long_rows()
    A, _ = make(csr, fmt)
    info = A.info()
    assert info["spmv_layout"] == 2 and info["adj_layout_fused"] == 2 and info["max_row_len"] > 900
    first = _outputs(A, csr)
    A.set_tuning(**info["tuning"])
    assert A.info() == info
    B, _ = make(csr, fmt, tuning=info["tuning"])
    assert B.info()["spmv_layout"] == 2 and B.info()["adj_layout_fused"] == 2 and B.info()["adj_layout_adjoint"] == 2
    for H in (A, B):  # the knobs in effect are the same, so the bits are
        for a, b in zip(first, _outputs(H, csr)):
            assert torch.equal(a, b)
        H.device_status()


def test_autotune_cache_hits(tmp_path):
    csr = _long_rows()
    cache = str(tmp_path / "autotune.json")
    x = _to(np.random.default_rng(4).uniform(0, 1, csr.ncols).astype(np.float32))
    A, _ = make(csr, "u16")
    assert A.autotune(x, mode="cached", purposes=("forward", "fused", "batched"), cache=cache)["source"] == "sweep"
    B, _ = make(csr, "u16")
    assert B.autotune(x, mode="cached", purposes=("forward", "fused", "batched"), cache=cache)["source"] == "cache"
    assert A.info()["tuning"] == B.info()["tuning"]


def test_a_refused_value_changes_nothing():
    csr = _long_rows()
    A, _ = make(csr, "u16")
    info = A.info()
    assert info["tuning"]["tile_rows"] != 512
    for bad in (dict(rg_tile_union=512), dict(adj_layout=2, rg_tile_union=256)):  # below the longest row
        with pytest.raises(dose.DoseError) as ei:
            A.set_tuning(tile_rows=512, **bad)
        assert ei.value.status == 1
        assert A.info() == info
    # at create an explicit value below the longest row leaves the layout out, or is refused with it asked for
    assert make(csr, "u16", tuning=dict(rg_tile_union=512))[0].info()["rg_groups"] == 0
    with pytest.raises(dose.DoseError) as ei:
        make(csr, "u16", tuning=dict(rg_tile_union=512, adj_layout=2))
    assert ei.value.status == 1


def test_reported_threads_per_cta():
    """adj_block_*: every warp of the launch, those of the rows without entries too."""
    for csr in (_long_rows(), dosegen.generate(dosegen.TINY)):
        A, _ = make(csr, "u16", tuning=dict(rg_warps=5))
        info = A.info()
        assert info["rg_warps_fused"] == 5
        assert info["adj_block_fused"] == 32 * (5 + 3) and info["adj_block_adjoint"] == 32 * 5


def test_no_memory_for_the_fused_copy_keeps_the_layout(monkeypatch):
    """Rows i, i + 64, ... see the same 25 columns, neighbours see others: the layout of
    the other calls stores 2.25 bytes an entry, the stored-row copy of the fused
    pass 10, the CSR columns 4.  With room for one more array of the columns' size the
    layout stays, and the fused pass runs on it."""
    n = 16000
    base = np.random.default_rng(5).permutation(1600).reshape(64, 25)
    base.sort(axis=1)
    col = base[np.arange(n) % 64].astype(np.uint32).reshape(-1)
    rp = (25 * np.arange(n + 1)).astype(np.uint32)
    csr = dosegen.CSR(n, 1600, rp, col, np.random.default_rng(6).uniform(0.1, 1.0, col.size))
    monkeypatch.setenv("DOSE_TEST_ALLOC_LIMIT", str(4 * ((csr.nnz + 3) // 4 * 4 + 16)))
    with pytest.raises(dose.DoseError) as ei:
        make(csr, "u16", tuning=dict(adj_layout=2))
    assert ei.value.status == 2
    A, enc = make(csr, "u16")
    monkeypatch.delenv("DOSE_TEST_ALLOC_LIMIT")
    info = A.info()
    assert info["rg_groups"] > 0 and info["spmv_layout"] == 2
    assert info["adj_layout_adjoint"] == 2 and info["adj_layout_fused"] == 2
    rng = np.random.default_rng(7)
    x = rng.uniform(0, 1, 1600).astype(np.float32)
    p = rng.uniform(0, 2, n).astype(np.float32)
    w = rng.uniform(0.5, 2.0, n).astype(np.float32)
    f, g, d = A.fwd_adj_quadratic(_to(x), _to(p), _to(w), want_d=True)
    fwd_check(d.cpu().numpy(), oracle.spmv(n, rp, col, enc.decoded, x))
    f_own, r_own = oracle.objective(d.cpu().numpy().astype(np.float64), p, w)
    assert abs(float(f.item()) - f_own) <= 1e-12 * f_own
    adj_check(g.cpu().numpy(), oracle.spmv_t(n, 1600, rp, col, enc.decoded, r_own),
              oracle.abs_spmv_t(n, 1600, rp, col, enc.decoded, r_own))
    A.device_status()


@pytest.mark.parametrize("long_rows", [True, False])
def test_knobs_that_do_not_fit_change_nothing(monkeypatch, long_rows):
    """dose_set_tuning without memory for the new deals or schedules (the limit lets
    some of them through): the handle reports and computes what it did before."""
    csr = _long_rows() if long_rows else dosegen.generate(dosegen.TINY)
    A, _ = make(csr, "u16")
    info, first = A.info(), _outputs(A, csr)
    for limit in (15, 1000, 3000):
        monkeypatch.setenv("DOSE_TEST_ALLOC_LIMIT", str(limit))
        with pytest.raises(dose.DoseError) as ei:
            A.set_tuning(rg_warps=2, adj_tile_nnz=512, tile_nnz=2048)
        monkeypatch.delenv("DOSE_TEST_ALLOC_LIMIT")
        assert ei.value.status == 2
        assert A.info() == info
        for a, b in zip(first, _outputs(A, csr)):
            assert torch.equal(a, b)
    A.device_status()
