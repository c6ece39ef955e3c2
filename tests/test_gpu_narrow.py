"""Networks whose weights are small beside their parts (widths of 8 to 16, parts of 10^5 rows and more), in contexts whose
scratch is limited to what the call says it needs.  Against the fp64 oracle."""
import re

import numpy as np
import pytest
import torch

import oracle
from paper_2305_09887_b200 import binding, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def util():
    import gpu_util
    return gpu_util


def _needed(dims, n, variant=(0, 0, 0), record=False):
    """Bytes of scratch that a call with one part of n rows says it needs."""
    c = binding.Context(0)
    c.set_workspace_limit(4096)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    X, y = torch.zeros(n, dims[0], device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    params = torch.zeros(1, binding.param_count(dims, variant), device="cuda")
    taps = (torch.empty(n * sum(a + b for a, b in zip(dims[:-1], dims[1:])), device="cuda"), None, 0) if record else None
    with pytest.raises(binding.RtmaError) as e:
        c.local_steps(dims, 0.1, 1, [0, n], [0, 0], rowptr, torch.empty(0, dtype=torch.int32, device="cuda"), X, y, params, 1, variant=variant,
                      taps=taps)
    c.close()
    return int(re.search(r"need (\d+) bytes of scratch", str(e.value)).group(1))


def _workload(n, degree, dims, variant, M=1):
    g = inputs.uniform_graph(n, n * degree // 2, 41)
    X, y = inputs.normal_features(n, dims[0], 42), inputs.uniform_labels(n, dims[-1], 43)
    rng = np.random.default_rng(44)
    p0 = oracle.variant_init_params(variant, dims, 45)
    p0 = (p0 + 0.02 * rng.standard_normal(p0.size)).astype(np.float32)
    return inputs.Workload("narrow", g, X, y, dims, M=M, K=2, R=1, lr=0.01, partition_seed=46, params0=p0)


# Layer Normalization and PReLU: their partial sums leave no room that other lists could lie in
@pytest.mark.parametrize("n, dims, variant", [(1_000_000, (8, 8, 2), (0, 1, 1)), (400_000, (3, 4, 2), (0, 1, 0)), (2_500_000, (16, 16, 5), (1, 1, 1))])
def test_a_call_on_a_large_part_fits_the_scratch_it_asks_for(util, monkeypatch, n, dims, variant):
    w = _workload(n, 4, dims, variant)
    c = binding.Context(0)
    c.set_workspace_limit(_needed(dims, n, variant, record=True))  # check_one_step records the activations
    monkeypatch.setattr(util, "_ctx", c)
    util.check_one_step(w, variant=variant)
    c.check()
    c.close()


def test_long_rows_listed_or_searched_for_give_the_same_bits(util):
    # tensor-core tiles forced on a graph without neighbourhoods: nearly all of 72,000 rows have more entries outside their windows than
    # are listed, two of them hundreds.  A context that has no room to list such rows, one that has, and one whose arena a call grew
    n, dims = 72_000, (16, 16, 5)
    w = _workload(n, 9, dims, (0, 0, 0))
    g = w.graph
    rng = np.random.default_rng(47)
    rows, cols = np.repeat(np.arange(n), np.diff(g.rowptr)), g.col.astype(np.int64)
    hubs = [(v, rng.permutation(n)[:size]) for v, size in ((5, 500), (n - 3, 320))]
    u = np.concatenate([rows] + [np.full(x.size, v) for v, x in hubs] + [x for _, x in hubs])
    v = np.concatenate([cols] + [x for _, x in hubs] + [np.full(x.size, h) for h, x in hubs])
    key = np.unique((u * n + v)[u != v])
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=rowptr[1:])
    col = util.dev((key % n).astype(np.int32))

    def run(workspace_bytes, limit):
        c = binding.Context(0, workspace_bytes)
        c.set_workspace_limit(limit)
        c.set_dense_aggregation(2)
        params = util.dev(w.params0[None])
        c.local_steps(dims, 0.1, 1, [0, n], [0, int(rowptr[-1])], util.dev(rowptr), col, util.dev(w.X), util.dev(w.y), params, 3)
        c.check()
        out, size = params.cpu().numpy()[0], c.workspace_bytes
        c.close()
        return out, size

    need = _needed(dims, n)
    searched, size = run(0, need)
    assert size <= need
    listed, size = run(need + 4 * n + 4096, 0)
    assert size == need + 4 * n + 4096
    grown, _ = run(0, 0)
    assert np.array_equal(searched, listed) and np.array_equal(searched, grown)
    want, _ = oracle.local_steps_variant((0, 0, 0), dims, 0.1, rowptr, (key % n).astype(np.int32), w.X.astype(np.float64), w.y,
                                         w.params0.astype(np.float64), 3)
    assert util.rel_err(searched, want) <= util.TOL_PARAM


@pytest.mark.parametrize("dims, M", [((10, 33, 3), 1), ((10, 70, 33), 2), ((20, 5), 1)])
def test_as_many_chunks_as_a_part_may_have_of_an_odd_width(util, dims, M):
    # the padded rows of the partial sums do not fit then: they follow one another, at addresses that no bulk-tensor store can take
    n = 140_000
    sums = [(c * (2 * a + 1), b) for c, a, b in zip(binding.selftest_chunks(dims, n // M, M), dims[:-1], dims[1:])]
    assert max(rows * -(-b // 4) * 4 for rows, b in sums) > 64 * max((2 * a + 1) * b for a, b in zip(dims[:-1], dims[1:]))
    w = _workload(n, 3, dims, (0, 0, 0), M)
    got, want = util.check_one_step(w)
    util.check_k_steps_and_average(w, got, want, 2)


def test_linear_decoder_on_many_pairs(util):
    import test_gpu_link as tl
    w = _workload(30_000, 8, (24, 40, 40), (0, 0, 0))
    assert binding.selftest_chunks(w.dims, 131_072, ddims=(40, 1))[-1] == 64
    tl._check_link(util, w, (0, 1, 1), (40, 1), per_part=65_536, K=2)
