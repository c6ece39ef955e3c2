"""The range-checked build of the library (-DRTMA_BOUNDS, librtma_checked.so): every index a kernel
takes from the caller's data is checked before it addresses memory; an index out of range is recorded,
the access is skipped, and the next rtma_check returns RTMA_ERR_BOUNDS.  It stands in for a memory
checker: on healthy inputs it must give the ordinary build's result bit for bit and report nothing; on
inputs with a bad index it must say which, without touching memory out of range.
"""
import numpy as np
import pytest
import torch

import gpu_util
from paper_2305_09887_b200 import binding, inputs

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _whole_path(c, w):
    g = w.graph
    part_id, part_offsets, perm, local_id = c.partition(g.n, None, w.partition_seed, w.M)
    rowptr_out, col_out, edge_offsets, kept_cut, edge_host = c.build_induced_csr(
        _dev(g.rowptr), _dev(g.col), w.M, part_id, part_offsets, perm, local_id)
    yp = c.gather_rows(_dev(w.y), perm)
    params = _dev(np.tile(w.params0, (w.M, 1)))
    loss = torch.zeros(w.M, w.K, dtype=torch.float32, device="cuda")
    c.local_steps(w.dims, w.lr, w.M, part_offsets.cpu().tolist(), edge_host, rowptr_out, col_out, _dev(w.X), yp, params,
                  w.K, loss_out=loss, perm=perm)
    c.aggregate(params)
    c.check()
    return perm, rowptr_out, col_out, params, loss


def test_checked_build_agrees_with_the_ordinary_one(tiny_workload):
    lib = binding.load_library(checked=True)
    assert lib.rtma_bounds_checked() == 1 and binding.load_library().rtma_bounds_checked() == 0
    for w in (tiny_workload, inputs.medium(0.03)):
        plain = _whole_path(binding.Context(0), w)
        checked = _whole_path(binding.Context(0, checked=True), w)
        for a, b in zip(plain, checked):
            assert torch.equal(a, b)


def test_checked_build_reports_a_column_id_out_of_range(tiny_workload):
    w = tiny_workload
    g = w.graph
    c = binding.Context(0, checked=True)
    part_id, part_offsets, perm, local_id = c.partition(g.n, None, w.partition_seed, w.M)
    col = g.col.copy()
    col[123] = g.n + 5                                   # one entry points past the last node
    with pytest.raises(binding.RtmaError, match="column id of the input graph 2005 outside"):
        c.build_induced_csr(_dev(g.rowptr), _dev(col), w.M, part_id, part_offsets, perm, local_id)
        c.check()
    c.check()                                            # reported once; the context stays usable
    good = c.build_induced_csr(_dev(g.rowptr), _dev(g.col), w.M, part_id, part_offsets, perm, local_id)
    c.check()
    assert int(good[3][0]) + int(good[3][1]) == g.num_entries


def test_checked_build_reports_a_label_out_of_range(tiny_workload):
    w = tiny_workload
    g = w.graph
    c = binding.Context(0, checked=True)
    part_id, part_offsets, perm, local_id = c.partition(g.n, None, w.partition_seed, w.M)
    rowptr_out, col_out, edge_offsets, kept_cut, edge_host = c.build_induced_csr(
        _dev(g.rowptr), _dev(g.col), w.M, part_id, part_offsets, perm, local_id)
    y = w.y.copy()
    y[77] = w.dims[-1]                                   # one class id past the last class
    yp = c.gather_rows(_dev(y), perm)
    params = _dev(np.tile(w.params0, (w.M, 1)))
    c.local_steps(w.dims, w.lr, w.M, part_offsets.cpu().tolist(), edge_host, rowptr_out, col_out, _dev(w.X), yp, params, 1,
                  perm=perm)
    with pytest.raises(binding.RtmaError, match="label 8 outside"):
        c.check()


def test_a_row_with_a_bad_permutation_entry_counts_as_zeros(tiny_workload):
    w = tiny_workload
    g = w.graph
    c = binding.Context(0, checked=True)
    gpu_util.fill_scratch_with_nan(c, g)
    part_id, part_offsets, perm, local_id = c.partition(g.n, None, w.partition_seed, w.M)
    rowptr_out, col_out, _, _, edge_host = c.build_induced_csr(_dev(g.rowptr), _dev(g.col), w.M, part_id, part_offsets, perm, local_id)
    yp = c.gather_rows(_dev(w.y), perm)
    part_host = part_offsets.cpu().tolist()

    def steps(X, order):
        params = _dev(np.tile(w.params0, (w.M, 1)))
        c.local_steps(w.dims, w.lr, w.M, part_host, edge_host, rowptr_out, col_out, X, yp, params, 2, perm=order)
        return params

    bad = perm.clone()
    bad[900] = g.n + 3
    got = steps(_dev(w.X), bad)
    with pytest.raises(binding.RtmaError, match=f"permutation entry {g.n + 3} outside"):
        c.check()
    X = _dev(w.X)
    X[int(perm[900])] = 0.0
    want = steps(X, perm)
    c.check()
    assert torch.equal(got, want)


def test_a_bad_pair_counts_as_zeros(tiny_workload):
    w = tiny_workload
    g = w.graph
    c = binding.Context(0, checked=True)
    gpu_util.fill_scratch_with_nan(c, g)
    part_id, part_offsets, perm, local_id = c.partition(g.n, None, w.partition_seed, 2)
    rowptr_out, col_out, _, _, edge_host = c.build_induced_csr(_dev(g.rowptr), _dev(g.col), 2, part_id, part_offsets, perm, local_id)
    part_host = part_offsets.cpu().tolist()
    dims, ddims = (64, 40, 24), (24, 16, 1)
    rng = np.random.default_rng(5)
    pu, pv = (rng.integers(0, min(part_host[1], g.n - part_host[1]), size=180).astype(np.int32) for _ in range(2))
    pu[77] = 1 << 20
    params = _dev(np.tile(rng.normal(size=binding.link_param_count(dims, ddims)).astype(np.float32) * 0.1, (2, 1)))
    c.link_steps(dims, ddims, 0.05, 2, part_host, edge_host, rowptr_out, col_out, c.gather_rows(_dev(w.X), perm), [0, 101, 180],
                 _dev(pu), _dev(pv), _dev((rng.random(180) < 0.5).astype(np.int32)), params, 2)
    with pytest.raises(binding.RtmaError, match=f"{1 << 20} outside"):
        c.check()
    assert torch.isfinite(params).all()
