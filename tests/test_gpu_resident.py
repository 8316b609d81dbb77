"""GPU parity of ComplEx on rows that stay in shared memory: chunks of 64 dimensions and their remainders, every alignment of a row's second
half, one to 32 rows per data point, clusters for few data points and for wide rows; both sides of the last sizes that fit a block, a
cluster of two and one of four, and the streamed kernel beyond them."""
import numpy as np
import pytest
import torch

import paper_2002_00655_b200 as ps
from tests.test_gpu_sorted import EPS, LR, ada_rows, check, check_no_op, on_gpu, triples
from tests.util import close, make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n_neg", [(129, 10), (130, 0), (132, 20), (191, 29), (320, 10), (578, 13), (832, 29), (834, 29), (1001, 4), (1216, 20),
                                       (2176, 10), (2178, 10), (66, 11), (100, 29), (127, 20), (2501, 20), (4098, 10), (8704, 10), (9000, 10)])
@pytest.mark.parametrize("few", [2, 75, 0])
def test_complex_rows_kept_in_shared_memory(dim, n_neg, few):
    rng = np.random.default_rng(dim + few)
    n = few or 8192 // (3 + n_neg) + 5                          # 0: as many as take a sort
    E, R = (40, 3) if few else (n, 7)                           # (few entities: the same one in several places of a data point)
    K = E + R
    g, o = make_pair(K, 4 * dim, rows=ada_rows(rng, K, 4 * dim), max_batch_keys=(3 + n_neg) * n)
    ps.ps_set_pipelining(g.h, True)
    batches = [triples(rng, n, n_neg, E, R) for _ in range(2)]
    gpu = [on_gpu(b) for b in batches]
    torch.cuda.synchronize()
    for b, d in zip(batches, gpu):
        ps.ps_step_kge(g.h, *d, n_neg, E, dim, LR, EPS, g.loss)
        o.step_kge(*b, E, dim, LR, EPS)
    check(g, o, "complex")
    bad = [x.copy() for x in batches[0]]
    bad[2][-1] = E
    d = on_gpu(bad)
    torch.cuda.synchronize()
    check_no_op(g, o, lambda: ps.ps_step_kge(g.h, *d, n_neg, E, dim, LR, EPS, g.loss), "an object out of range")


# The last dimension that a block, a cluster of two and one of four take, and the next, by the number of negatives (launch_resident's sums
# for 227 KB of shared memory and the fewest warps per SM); beyond the last the rows are streamed.
@pytest.mark.parametrize("dim,n_neg", [(2112, 10), (2116, 10), (4224, 10), (4228, 10), (8448, 10), (8452, 10), (2047, 10), (2049, 10), (3838, 10),
                                       (3842, 10), (7679, 10), (7681, 10), (7682, 10), (1152, 20), (1156, 20), (2304, 20), (2308, 20), (4608, 20),
                                       (4612, 20), (4095, 20), (4097, 20), (4102, 20), (832, 29), (836, 29), (1536, 29), (1540, 29), (3072, 29),
                                       (3076, 29), (3071, 29), (3074, 29), (3077, 29), (4032, 4), (4036, 4), (8064, 4), (8068, 4), (15360, 4),
                                       (15364, 4), (14335, 4), (14337, 4), (14338, 4), (1920, 11), (1924, 11), (7180, 11), (3702, 25)])
@pytest.mark.parametrize("n", [2, 75])
def test_complex_rows_around_the_last_sizes_that_fit(dim, n_neg, n):
    """Two data points: no sort (odd dimensions: finished rows, streamed); 75: with a sort and rows updated in place."""
    test_complex_rows_kept_in_shared_memory(dim, n_neg, n)


@pytest.mark.parametrize("dim,n_neg,n", [(2116, 10, 150), (4097, 20, 75), (300, 29, 60), (577, 20, 40)])
def test_complex_clusters_from_host_batches_and_graphs(dim, n_neg, n):
    """The rows of ordered calls, bit for bit: batches from pinned host memory, several in flight; a graph of two steps, replayed."""
    rng = np.random.default_rng(dim)
    E, R = 2 * n, 5
    rows = ada_rows(rng, E + R, 4 * dim)
    a, h, c = (make_pair(E + R, 4 * dim, rows=rows, max_batch_keys=(3 + n_neg) * n)[0] for _ in range(3))
    for s in (h, c):
        ps.ps_set_pipelining(s.h, True)
    ps.ps_set_host_overlap(h.h, True)
    batches = [triples(rng, n, n_neg, E, R) for _ in range(4)]
    pinned = [[torch.from_numpy(x.view(np.int32) if x.dtype == np.uint32 else x).pin_memory() for x in b] for b in batches]
    gpu = [on_gpu(b) for b in batches]
    words = torch.zeros(4, dtype=torch.float64).pin_memory()
    torch.cuda.synchronize()
    step = lambda s, i: ps.ps_step_kge(s.h, *gpu[i], n_neg, E, dim, LR, EPS, s.loss)
    for i in range(4):
        ps.ps_step_kge_host(h.h, *pinned[i], n_neg, E, dim, LR, EPS, h.loss, words[i:i + 1])
    want = []
    for i in range(4):
        step(a, i)
        a.sync()
        want.append(float(a.loss.cpu()[0]))
    h.sync()
    assert torch.equal(a.export(table=False)[0], h.export(table=False)[0]) and words.tolist() == want
    step(c, 0)
    torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(stream):
        graph.capture_begin(capture_error_mode="thread_local")
        step(c, 1)
        step(c, 2)
        graph.capture_end()
    graph.replay()
    torch.cuda.synchronize()
    step(c, 3)
    assert c.sync() == ps.PS_OK
    assert torch.equal(a.export(table=False)[0], c.export(table=False)[0]) and float(c.loss.cpu()[0]) == want[-1]


@pytest.mark.parametrize("dim,n_neg,n", [(100, 10, 60), (130, 10, 30), (577, 4, 200), (2116, 10, 75), (2049, 10, 75), (8452, 10, 40)])
def test_complex_rows_that_are_not_finite(dim, n_neg, n):
    """Rows with an infinite or no number in one dimension, in every entity's place; signs such that no sum of a score's terms meets
    infinities of both.  In all other dimensions the oracle's rows, finite or not; in that one nothing finite that is not so in the oracle."""
    rng = np.random.default_rng(dim)
    E, R = 40 * n, 5
    rows = np.abs(ada_rows(rng, E + R, 4 * dim)) + np.float32(0.01)
    rows[:4, dim - 1] = np.inf                                  # Re, for the subject's place
    rows[4:8, 2 * dim - 1] = np.inf                             # Im, for the object's
    rows[8:12, 0] = np.nan
    g, o = make_pair(E + R, 4 * dim, rows=rows, max_batch_keys=(3 + n_neg) * n)
    s, r, t, ne, ns = triples(rng, n, n_neg, E, R)
    s, t, ne = (x % np.uint32(E - 12) + np.uint32(12) for x in (s, t, ne))
    r = r % np.uint32(R - 1) + np.uint32(1)
    r[:12] = 0
    s[:2], t[2:4], ne[4:8, 0], ns[4:8, 0] = (0, 1), (4, 5), (2, 3, 6, 7), (0, 0, 1, 1)
    s[8], t[9], ne[10:12, 1] = 8, 9, (10, 11)
    batch = (s, r, t, ne, ns)
    ps.ps_step_kge(g.h, *on_gpu(batch), n_neg, E, dim, LR, EPS, g.loss)
    o.step_kge(*batch, E, dim, LR, EPS)
    g.sync()
    got = g.export(table=False)[0].numpy()
    ok, fine = np.isfinite(o.rows), np.isfinite(got)
    assert 0 < (~ok).sum() < ok.size // 2 and not (fine & ~ok).any()
    special = np.isin(np.arange(4 * dim) % dim, (0, dim - 1))
    assert (fine[:, ~special] == ok[:, ~special]).all()
    assert close(got[fine], o.rows[fine]).all()
