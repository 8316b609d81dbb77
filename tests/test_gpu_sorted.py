"""GPU parity of the steps on their sorted kernels (more than 8,192 key occurrences): rows updated in place in pipelined mode,
runs of one key of every length, bad indexes, host batches and graph replays at sizes where a sort is taken."""
import numpy as np
import pytest
import torch

import paper_2002_00655_b200 as ps
from tests.util import close, compare_state, dev, make_pair

pytestmark = pytest.mark.gpu
LR, EPS = 0.1, 1e-8
SMALL = 8192                                    # key occurrences up to which a call takes no sort


def u32(a):
    return np.ascontiguousarray(a, dtype=np.uint32)


def triples(rng, n, n_neg, E, R):
    """Entities with a few frequent ones and many that occur once."""
    pick = lambda *shape: u32(np.where(rng.random(shape) < 0.2, rng.integers(0, 30, size=shape), rng.integers(0, E, size=shape)))
    return pick(n), u32(rng.integers(0, R, size=n)), pick(n), pick(n, n_neg), rng.integers(0, 2, size=(n, n_neg)).astype(np.uint8)


def on_gpu(batch):
    return [dev(x, torch.uint8 if x.dtype == np.uint8 else torch.float32 if x.dtype == np.float32 else torch.int32) for x in batch]


def ada_rows(rng, K, L):
    rows = rng.normal(0, 0.3, size=(K, L)).astype(np.float32)
    rows[:, L // 2:] = rows[:, L // 2:] ** 2 + 0.01             # accumulators some way into training
    return rows


def loss_of(g):
    return float(g.loss.cpu()[0])


def check(g, o, what):
    g.sync()
    compare_state(g, o, what=what)
    assert close(loss_of(g), o.loss[0]), (what, loss_of(g), o.loss[0])


def check_no_op(g, o, call, what):
    before = loss_of(g), g.export()[0]
    call()
    assert g.sync(check=False) == ps.PS_ERR_KEY_RANGE, what
    assert torch.equal(g.export()[0], before[1]) and loss_of(g) == before[0], what


@pytest.mark.parametrize("pipelined", [False, True])
@pytest.mark.parametrize("dim,n_neg", [(1, 10), (33, 3), (33, 29), (100, 10), (127, 20), (128, 3), (128, 29), (130, 3), (257, 12)])
def test_complex_steps_with_a_sort(dim, n_neg, pipelined):
    rng = np.random.default_rng(dim * 31 + n_neg)
    n, E, R = SMALL // (3 + n_neg) + 37, 6_000, 7
    rows = ada_rows(rng, E + R, 4 * dim)
    g, o = make_pair(E + R, 4 * dim, 2, rows=rows, max_batch_keys=(3 + n_neg) * n)
    ps.ps_set_pipelining(g.h, pipelined)
    batch = triples(rng, n, n_neg, E, R)
    d = on_gpu(batch)
    torch.cuda.synchronize()
    ps.ps_step_kge(g.h, *d, n_neg, E, dim, LR, EPS, g.loss)
    o.step_kge(*batch, E, dim, LR, EPS)
    check(g, o, "complex")
    for which, bad in ((0, E), (1, R), (2, E + R), (3, E)):     # each index out of range in turn, late in the batch
        b = [x.copy() for x in batch]
        b[which].reshape(-1)[-2] = bad
        d = on_gpu(b)
        torch.cuda.synchronize()
        check_no_op(g, o, lambda: ps.ps_step_kge(g.h, *d, n_neg, E, dim, LR, EPS, g.loss), f"complex, bad index in array {which}")


@pytest.mark.parametrize("pipelined", [False, True])
@pytest.mark.parametrize("row,window,n_neg", [(8, 2, 3), (128, 1, 5), (132, 3, 0), (256, 2, 3), (260, 5, 3), (300, 5, 3), (384, 4, 2),
                                              (388, 2, 6), (512, 3, 2)])
def test_skip_gram_steps_with_a_sort(row, window, n_neg, pipelined):
    rng = np.random.default_rng(row + window)
    slots = 1 + 2 * window * (1 + n_neg)
    n, V = SMALL // slots + 61, 4_000
    T = n + 3                                                    # clipped windows at both ends of the stream
    occ = n * slots
    rows = rng.normal(0, 0.1, size=(2 * V, row)).astype(np.float32)
    word = lambda *shape: u32(np.where(rng.random(shape) < 0.3, rng.integers(0, 20, size=shape), rng.integers(0, V, size=shape)))
    tok, neg = word(T), word(n * 2 * window, max(n_neg, 1))
    g, o = make_pair(2 * V, row, rows=rows, max_batch_keys=max(occ, 3 * n))
    ps.ps_set_pipelining(g.h, pipelined)
    d = on_gpu((tok, neg))
    torch.cuda.synchronize()
    ps.ps_step_sgns(g.h, d[0], 0, n, window, d[1], n_neg, V, 0.01, g.loss)
    o.step_sgns(tok, 0, n, window, neg[:, :n_neg], n_neg, V, 0.01)
    check(g, o, "skip-gram")
    bad = tok.copy()
    bad[n // 2] = V
    d = on_gpu((bad, neg))
    torch.cuda.synchronize()
    check_no_op(g, o, lambda: ps.ps_step_sgns(g.h, d[0], 0, n, window, d[1], n_neg, V, 0.01, g.loss), "skip-gram, bad word")


@pytest.mark.parametrize("pipelined", [False, True])
def test_bad_indexes_of_sorted_matrix_and_rescal_steps(pipelined):
    rng = np.random.default_rng(5)
    R, C, n = 3_000, 500, 5_000
    g, o = make_pair(R + C, 20, max_batch_keys=2 * n)
    ps.ps_set_pipelining(g.h, pipelined)
    for which, bad in ((0, R), (1, C)):
        a = [u32(rng.integers(0, R, size=n)), u32(rng.integers(0, C, size=n)), rng.normal(size=n).astype(np.float32)]
        a[which][n - 3] = bad
        d = on_gpu(a)
        torch.cuda.synchronize()
        check_no_op(g, o, lambda: ps.ps_step_mf(g.h, *d, R, 0.01, 0.05, g.loss), "matrix factorization")
    E, R, dim, n_neg, n = 2_000, 9, 20, 6, 700
    g, o = make_pair(E + R * dim, 2 * dim, rows=ada_rows(rng, E + R * dim, 2 * dim), max_batch_keys=(2 + n_neg + dim) * n)
    ps.ps_set_pipelining(g.h, pipelined)
    for which, bad in ((0, E), (1, R), (2, E), (3, E)):
        b = list(triples(rng, n, n_neg, E, R))
        b[which].reshape(-1)[-2] = bad
        d = on_gpu(b)
        torch.cuda.synchronize()
        check_no_op(g, o, lambda: ps.ps_step_rescal(g.h, *d, n_neg, E, dim, LR, EPS, g.loss), f"RESCAL, array {which}")


@pytest.mark.parametrize("pipelined", [False, True])
@pytest.mark.parametrize("dim", [12, 33, 100, 150])
def test_adagrad_runs_of_every_length(dim, pipelined):
    """Subjects that occur 1, 2, 11, 12, 39, 40, 143, 144, 240, 1,000 and 3,000 times (added by a warp, by a block, in pieces by
    several), relations of a third and of a single data point; everything else occurs once."""
    rng = np.random.default_rng(dim)
    runs = [1, 2, 3, 11, 12, 13, 39, 40, 41, 143, 144, 145, 240, 1_000, 3_000]
    s = np.repeat(np.arange(len(runs)), runs)
    n, n_neg = len(s), 1
    rng.shuffle(s)
    E, R = len(runs) + 2 * n, 4
    fresh = len(runs) + rng.permutation(2 * n)
    r = rng.integers(0, 3, size=n)
    r[7] = 3
    batch = u32(s), u32(r), u32(fresh[:n]), u32(fresh[n:].reshape(n, 1)), rng.integers(0, 2, size=(n, 1)).astype(np.uint8)
    g, o = make_pair(E + R, 4 * dim, rows=ada_rows(rng, E + R, 4 * dim), max_batch_keys=4 * n)
    ps.ps_set_pipelining(g.h, pipelined)
    d = on_gpu(batch)
    torch.cuda.synchronize()
    ps.ps_step_kge(g.h, *d, n_neg, E, dim, LR, EPS, g.loss)
    o.step_kge(*batch, E, dim, LR, EPS)
    check(g, o, "runs")


@pytest.mark.parametrize("d,rels,n", [(4, 1, 2_500), (12, 2, 1_500), (64, 1, 700), (100, 1, 1_200), (128, 3, 500)])
def test_rescal_relations_of_many_chunks(d, rels, n):
    """Relations whose data points are cut into one to 150 chunks, summed in groups."""
    rng = np.random.default_rng(d)
    E, n_neg = 9_000, 4
    K = E + rels * d
    g, o = make_pair(K, 2 * d, rows=ada_rows(rng, K, 2 * d), max_batch_keys=(2 + n_neg + d) * n)
    batch = triples(rng, n, n_neg, E, rels)
    ps.ps_step_rescal(g.h, *on_gpu(batch), n_neg, E, d, 0.02, EPS, g.loss)
    o.step_rescal(*batch, E, d, 0.02, EPS)
    check(g, o, "RESCAL chunks")


def test_overlapped_host_steps_with_a_sort_leave_the_rows_of_the_device_calls():
    """ComplEx, skip-gram and matrix factorization from pinned host memory, several calls in flight: rows and losses bit for bit."""
    rng = np.random.default_rng(11)
    E, R, dim, n_neg, n = 3_000, 11, 24, 10, 700
    V, row, window, q, m = 900, 264, 2, 3, 600
    C, rank, cells = 400, 36, 5_000
    kge = [triples(rng, n, n_neg, E, R) for _ in range(5)]
    sg = [(u32(rng.integers(0, V, size=m + 2 * window)), u32(rng.integers(0, V, size=(m * 2 * window, q)))) for _ in range(5)]
    mf = [(u32(rng.integers(0, E, size=cells)), u32(rng.integers(0, C, size=cells)), rng.normal(size=cells).astype(np.float32)) for _ in range(5)]
    shapes = [(E + R, 4 * dim, (3 + n_neg) * n), (2 * V, row, m * (1 + 2 * window * (1 + q))), (E + C, rank, 2 * cells)]
    stores = []
    for K, L, occ in shapes:
        rows = np.abs(rng.normal(0, 0.1, size=(K, L))).astype(np.float32) + 0.01
        (a, _), (b, _) = (make_pair(K, L, rows=rows, max_batch_keys=occ) for _ in range(2))
        ps.ps_set_pipelining(b.h, True)
        ps.ps_set_host_overlap(b.h, True)
        stores.append((a, b))
    pin = lambda batch: [torch.from_numpy(x.view(np.int32) if x.dtype == np.uint32 else x).pin_memory() for x in batch]
    kge_p, sg_p, mf_p = ([pin(b) for b in x] for x in (kge, sg, mf))
    words = torch.zeros((3, 5), dtype=torch.float64).pin_memory()
    for i in range(5):
        ps.ps_step_kge_host(stores[0][1].h, *kge_p[i], n_neg, E, dim, LR, EPS, stores[0][1].loss, words[0, i:i + 1])
        ps.ps_step_sgns_host(stores[1][1].h, sg_p[i][0], 0, window, m, m + 2 * window, window, sg_p[i][1], q, V, 0.01, stores[1][1].loss,
                             words[1, i:i + 1])
        ps.ps_step_mf_host(stores[2][1].h, *mf_p[i], E, 0.01, 0.05, stores[2][1].loss, words[2, i:i + 1])
    want = torch.zeros_like(words)
    for i in range(5):
        a = [s[0] for s in stores]
        ps.ps_step_kge(a[0].h, *on_gpu(kge[i]), n_neg, E, dim, LR, EPS, a[0].loss)
        t = on_gpu(sg[i])
        ps.ps_step_sgns(a[1].h, t[0], window, m, window, t[1], q, V, 0.01, a[1].loss)
        ps.ps_step_mf(a[2].h, *on_gpu(mf[i]), E, 0.01, 0.05, a[2].loss)
        for j in range(3):
            a[j].sync()
            want[j, i] = loss_of(a[j])
    for a, b in stores:
        b.sync()
        assert torch.equal(a.export(table=False)[0], b.export(table=False)[0])
    assert torch.equal(words, want)


@pytest.mark.parametrize("pipelined", [False, True])
@pytest.mark.parametrize("n", [40, 900])
def test_complex_steps_replayed_from_a_graph(n, pipelined):
    """Captured once, replayed three times: the rows of the same calls made one by one; without and with a sort."""
    rng = np.random.default_rng(n)
    E, R, dim, n_neg = 1_500, 5, 20, 10
    rows = ada_rows(rng, E + R, 4 * dim)
    (a, _), (g, _) = (make_pair(E + R, 4 * dim, rows=rows, max_batch_keys=(3 + n_neg) * n) for _ in range(2))
    d = on_gpu(triples(rng, n, n_neg, E, R))
    for s in (a, g):
        ps.ps_set_pipelining(s.h, pipelined)
    step = lambda s: ps.ps_step_kge(s.h, *d, n_neg, E, dim, LR, EPS, s.loss)
    step(a); step(g)                                             # (kernels loaded, attributes set)
    torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(stream):
        graph.capture_begin(capture_error_mode="thread_local")
        step(g)
        step(g)
        graph.capture_end()
    for _ in range(3):
        graph.replay()
        step(a); step(a)
    torch.cuda.synchronize()
    assert a.sync() == g.sync() == ps.PS_OK
    assert torch.equal(a.export(table=False)[0], g.export(table=False)[0]) and loss_of(a) == loss_of(g)


@pytest.mark.parametrize("row", [4, 32, 36, 64, 68, 160, 164, 192, 196, 288, 320, 416, 448, 452])
def test_skip_gram_rows_whose_last_values_are_spread_over_the_lanes(row):
    """The reduction's last column block holds one, two or four values per lane: around the limits of each."""
    rng = np.random.default_rng(row)
    window, n_neg, V = 2, 3, 300
    n = SMALL // (1 + 2 * window * (1 + n_neg)) + 40
    g, o = make_pair(2 * V, row, rows=rng.normal(0, 0.1, size=(2 * V, row)).astype(np.float32), max_batch_keys=n * (1 + 2 * window * (1 + n_neg)))
    tok, neg = u32(rng.integers(0, V, size=n + 2 * window)), u32(rng.integers(0, V, size=(n * 2 * window, n_neg)))
    d = on_gpu((tok, neg))
    ps.ps_step_sgns(g.h, d[0], window, n, window, d[1], n_neg, V, 0.01, g.loss)
    o.step_sgns(tok, window, n, window, neg, n_neg, V, 0.01)
    check(g, o, "skip-gram")


@pytest.mark.parametrize("pipelined", [False, True])
@pytest.mark.parametrize("mode,dim,n", [("kge", 250, 492), ("kge", 250, 493), ("kge", 1001, 122), ("kge", 1001, 123), ("sgns", 300, 130),
                                        ("sgns", 300, 131), ("sgns", 512, 150)])
def test_wide_steps_on_either_side_of_the_sort(mode, dim, n, pipelined):
    """Few occurrences of wide rows: with and without a sort (1,600,000 dimensions or values of all occurrences), calls of both kinds
    one after the other."""
    rng = np.random.default_rng(dim + n)
    if mode == "kge":
        E, R, q = 900, 5, 10
        g, o = make_pair(E + R, 4 * dim, rows=ada_rows(rng, E + R, 4 * dim), max_batch_keys=(3 + q) * n)
        ps.ps_set_pipelining(g.h, pipelined)
        batches = [triples(rng, m, q, E, R) for m in (n, 9, n)]
        gpu = [on_gpu(b) for b in batches]
        torch.cuda.synchronize()
        for b, d in zip(batches, gpu):
            ps.ps_step_kge(g.h, *d, q, E, dim, LR, EPS, g.loss)
            o.step_kge(*b, E, dim, LR, EPS)
    else:
        V, window, q = 900, 5, 3
        g, o = make_pair(2 * V, dim, rows=rng.normal(0, 0.1, size=(2 * V, dim)).astype(np.float32), max_batch_keys=n * (1 + 2 * window * (1 + q)))
        ps.ps_set_pipelining(g.h, pipelined)
        batches = [(u32(rng.integers(0, V, size=m + 2 * window)), u32(rng.integers(0, V, size=(m * 2 * window, q))), m) for m in (n, 9, n)]
        gpu = [on_gpu(b[:2]) for b in batches]
        torch.cuda.synchronize()
        for (tok, neg, m), d in zip(batches, gpu):
            ps.ps_step_sgns(g.h, d[0], window, m, window, d[1], q, V, 0.01, g.loss)
            o.step_sgns(tok, window, m, window, neg, q, V, 0.01)
    check(g, o, mode)


@pytest.mark.parametrize("row,window,n_neg,n", [(400, 5, 3, 121), (400, 5, 3, 122), (512, 2, 2, 600), (300, 2, 5, 300), (320, 3, 3, 208), (260, 6, 3, 160),
                                                (512, 7, 7, 70)])
def test_wide_skip_gram_steps_by_slots_of_a_center(row, window, n_neg, n):
    """5,000 occurrences on either side, and centers of 13 to 113 slots: ordered and pipelined handles leave the oracle's rows, and
    the same bits."""
    rng = np.random.default_rng(row + n)
    V = 900
    rows = rng.normal(0, 0.1, size=(2 * V, row)).astype(np.float32)
    (g, o), (h, _) = (make_pair(2 * V, row, rows=rows, max_batch_keys=n * (1 + 2 * window * (1 + n_neg))) for _ in range(2))
    ps.ps_set_pipelining(h.h, True)
    for m in (n, 5, n):
        tok, neg = u32(rng.integers(0, V, size=m + 2 * window)), u32(rng.integers(0, V, size=(m * 2 * window, n_neg)))
        d = on_gpu((tok, neg))
        torch.cuda.synchronize()
        for s in (g, h):
            ps.ps_step_sgns(s.h, d[0], window, m, window, d[1], n_neg, V, 0.01, s.loss)
        o.step_sgns(tok, window, m, window, neg, n_neg, V, 0.01)
    check(g, o, "skip-gram")
    h.sync()
    assert torch.equal(g.export(table=False)[0], h.export(table=False)[0]) and loss_of(g) == loss_of(h)


@pytest.mark.parametrize("pipelined", [False, True])
@pytest.mark.parametrize("d,n_neg", [(64, 3), (68, 0), (128, 5)])
def test_rescal_blocks_that_take_several_pieces(d, n_neg, pipelined):
    """More pieces of relations than blocks: a block looks the next one up while it works on one."""
    rng = np.random.default_rng(d)
    E, rels, n = 2_500, 11, 4_000
    K = E + rels * d
    g, o = make_pair(K, 2 * d, rows=ada_rows(rng, K, 2 * d), max_batch_keys=(2 + n_neg + d) * n)
    ps.ps_set_pipelining(g.h, pipelined)
    batch = triples(rng, n, n_neg, E, rels)
    d_batch = on_gpu(batch)
    torch.cuda.synchronize()
    ps.ps_step_rescal(g.h, *d_batch, n_neg, E, d, 0.02, EPS, g.loss)
    o.step_rescal(*batch, E, d, 0.02, EPS)
    check(g, o, "RESCAL pieces")


@pytest.mark.parametrize("pipelined", [False, True])
def test_wide_skip_gram_steps_replayed_from_a_graph(pipelined):
    """Fewer than 8,192 occurrences, sorted for their width: captured once, replayed twice, against the same calls one by one."""
    rng = np.random.default_rng(5)
    V, row, window, n_neg, n = 700, 400, 5, 3, 130
    rows = rng.normal(0, 0.1, size=(2 * V, row)).astype(np.float32)
    (a, _), (g, _) = (make_pair(2 * V, row, rows=rows, max_batch_keys=n * (1 + 2 * window * (1 + n_neg))) for _ in range(2))
    d = on_gpu((u32(rng.integers(0, V, size=n + 2 * window)), u32(rng.integers(0, V, size=(n * 2 * window, n_neg)))))
    for s in (a, g):
        ps.ps_set_pipelining(s.h, pipelined)
    step = lambda s: ps.ps_step_sgns(s.h, d[0], window, n, window, d[1], n_neg, V, 0.01, s.loss)
    step(a); step(g)
    torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(stream):
        graph.capture_begin(capture_error_mode="thread_local")
        step(g)
        step(g)
        graph.capture_end()
    for _ in range(2):
        graph.replay()
        step(a); step(a)
    torch.cuda.synchronize()
    assert a.sync() == g.sync() == ps.PS_OK
    assert torch.equal(a.export(table=False)[0], g.export(table=False)[0]) and loss_of(a) == loss_of(g)
