"""Preparation and quality kernels on rows beyond what one thread handles, on ids too far apart for the packed
sort keys, and components of a graph too large for the component kernel's bitmap. Integers: exact equality."""
import numpy as np
import pytest

import oracle
from paper_1610_08128_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rcm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_08128_gb300 import build, rcm

    build.build()
    rcm.load()
    return rcm


def device(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def stars(sizes, seed):
    """Centres with the given numbers of neighbours, joined in a row, ids permuted."""
    src, dst, at = [], [], 0
    for i, s in enumerate(sizes):
        src += [np.full(s, at), np.array([at] if i else [], np.int64)]
        dst += [np.arange(at + 1, at + 1 + s), np.array([at - 1] if i else [], np.int64)]
        at += 1 + s
    g = synth.csr_from_edges(at, np.concatenate(src), np.concatenate(dst))
    return synth.permute(g, synth.random_permutation(at, seed))


LONG = {
    "around_64": lambda: stars(list(range(60, 70)) * 3, 1),
    "one_warp_of_them": lambda: stars([70] * 64, 2),
    "thousands": lambda: stars([3000, 1, 65, 9000, 7, 8, 9], 3),
    "hubs": lambda: synth.power_law(30_000, 10.0, 2.5, 4),
    "dense": lambda: synth.random_graph(700, 70_000, seed=5, connected=True),  # every row about 200
}


@pytest.mark.parametrize("name", list(LONG))
def test_bandwidth_and_profile(rcm, name):
    g = synth.shuffle_rows(LONG[name](), 6)
    rp, ci = device(g.rowptr), device(g.colidx)
    for perm in (synth.random_permutation(g.n, 7).astype(np.int32), np.arange(g.n, dtype=np.int32),
                 oracle.rcm(g.n, g.rowptr, g.colidx)):
        assert rcm.bandwidth_profile(rp, ci, device(perm)) == oracle.bandwidth_profile(g.n, g.rowptr, g.colidx, perm)


@pytest.mark.parametrize("at", [0, 31, 32, 63, 64, 65, 99])
@pytest.mark.parametrize("value", [-1, 2000, 1 << 30, -(1 << 31)])
def test_bad_entry_in_a_long_row(rcm, at, value):
    g = synth.csr_from_edges(2000, np.full(100, 1234), np.arange(100))
    colidx = g.colidx.copy()
    colidx[g.rowptr[1234] + at] = value
    rp, ci, perm = device(g.rowptr), device(colidx), torch.empty(2000, dtype=torch.int32, device="cuda")
    status = rcm.rcm_order(2000, rp, ci, perm)
    assert (status or rcm.rcm_stream_status()) == rcm.RCM_ERR_BAD_CSR
    goff = torch.tensor([0, 2000], device="cuda")
    status = rcm.rcm_order_batch(1, 2000, goff, rp, ci, perm)
    assert (status or rcm.rcm_stream_status()) == rcm.RCM_ERR_BAD_CSR


@pytest.mark.parametrize("rows", [64, 65, 100])
@pytest.mark.parametrize("last", [False, True])
def test_long_row_that_leaves_its_graph(rcm, rows, last):
    """Two graphs of 500 vertices, the first with a row of `rows` entries, one of them in the other graph."""
    g = synth.csr_from_edges(1000, np.full(rows, 400), np.arange(rows))
    row = g.colidx[g.rowptr[400]:g.rowptr[401]].copy()
    row[-1 if last else 0] = 700
    colidx = g.colidx.copy()
    colidx[g.rowptr[400]:g.rowptr[401]] = row
    perm = torch.empty(1000, dtype=torch.int32, device="cuda")
    goff = torch.tensor([0, 500, 1000], device="cuda")
    for ci, want in ((g.colidx, rcm.RCM_OK), (colidx, rcm.RCM_ERR_BAD_CSR)):
        status = rcm.rcm_order_batch(2, 1000, goff, device(g.rowptr), device(ci), perm)
        assert (status or rcm.rcm_stream_status()) == want


@pytest.mark.parametrize("apart", [-2, -1, 0, 1, 5000])
def test_ids_too_far_apart_for_packed_keys(rcm, apart):
    """Short rows whose neighbours' ids are 2^23 - 1, 2^23 and more from their own, on both sides."""
    far, m = (1 << 23) + apart, 30_000
    n = far + m
    rng = synth.rng_for([8, apart + 2])
    low = rng.integers(0, m, 40_000)
    g = synth.csr_from_edges(n, np.concatenate([np.arange(m), low]),
                             np.concatenate([np.arange(m) + far, rng.integers(n - m, n, 40_000)]))
    got = rcm.order(device(g.rowptr), device(g.colidx)).cpu().numpy()
    assert np.array_equal(got, oracle.rcm(g.n, g.rowptr, g.colidx))


def test_components_beyond_the_bitmap(rcm):
    """1.6M vertices in components of 200,000 and less, ordered by the component kernel without a bitmap."""
    b = synth.concat([synth.grid_fast((450, 450), seed=i) for i in range(7)] + [synth.grid_fast((50, 50, 50), seed=9)]
                     + [synth.grid((5, 9), seed=i) for i in range(400)])
    g = synth.permute(synth.Csr(b.n, b.rowptr, b.colidx), synth.random_permutation(b.n, 10))
    got, stats = rcm.order(device(g.rowptr), device(g.colidx), with_stats=True)
    assert stats["components"] == 408
    assert np.array_equal(got.cpu().numpy(), oracle.rcm(g.n, g.rowptr, g.colidx))


@pytest.mark.parametrize("last", [63, 99, 5000])
def test_bandwidth_with_the_most_entries(rcm, last):
    """2^31 - 1 stored entries: the offsets of the last rows are within a row's length of the largest int32."""
    free, _ = torch.cuda.mem_get_info()
    if free < 60 << 30:
        pytest.skip("needs 60 GB")
    n, nnz = 1 << 25, (1 << 31) - 1
    buf = torch.randint(0, n, (nnz + 1,), dtype=torch.int32, device="cuda")
    rowptr = torch.clamp(torch.arange(n + 1, device="cuda") * 64, max=nnz - last)
    rowptr[n] = nnz
    first = (nnz - last) // 64  # rows before this one have 64 entries
    buf[rowptr[n - 1]:nnz] = n - 2  # the last row reaches back by one, and by more in its last entry alone
    buf[nnz - 1] = 7
    beta = torch.arange(n, device="cuda")
    beta[:first] -= torch.minimum(beta[:first], buf[:64 * first].view(first, 64).amin(1).long())
    rest = buf[64 * first:nnz - last].long()
    beta[first:] = 0
    if len(rest):
        beta[first] = max(0, first - int(rest.min()))
    beta[n - 1] = n - 1 - 7
    got = rcm.bandwidth_profile(rowptr.int(), buf[:nnz], torch.arange(n, dtype=torch.int32, device="cuda"))
    assert got == (int(beta.max()), int(beta.sum()))
