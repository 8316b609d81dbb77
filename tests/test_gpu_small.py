"""GPU parity of the calls that are reduced without a sort (few key occurrences): sizes around the limits of that path,
hot keys that a whole block adds up, rows of one to many stretches of columns, bad indexes."""
import numpy as np
import pytest
import torch

import paper_2002_00655_b200 as ps
from synth import workloads as W
from tests.util import close, compare_state, dev, make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [4, 100, 132, 512, 520, 4100])
@pytest.mark.parametrize("n,hot", [(1, 0.0), (12, 0.0), (13, 1.0), (513, 0.3), (4096, 0.05), (8191, 0.9), (8192, 0.0), (8193, 0.0)])
def test_small_push_is_exact_on_integers(n, hot, L):
    K = 5000 if L < 500 else 700
    g, o = make_pair(K, L, 3, max_batch_keys=n)
    rng = np.random.default_rng(n + L)
    rows = rng.integers(-100, 100, size=(K, L)).astype(np.float32)
    g.set_all_rows(torch.from_numpy(rows))
    o.set_rows(np.arange(K), rows)
    keys = rng.integers(0, K, size=n)
    keys[rng.random(n) < hot] = K // 2
    keys[-1] = K - 1
    upd = rng.integers(-4, 5, size=(n, L)).astype(np.float32)     # integers: sums are exact in any order
    g.push(dev(keys), dev(upd))
    o.push(keys, upd)
    g.sync()
    compare_state(g, o, exact_rows=True, what="small push")
    if n > 1:
        keys[n // 2] = K                                           # one bad key: the call changes nothing
        g.push(dev(keys), dev(upd))
        assert g.sync(check=False) == ps.PS_ERR_KEY_RANGE
        compare_state(g, o, exact_rows=True, what="small push with a bad key")


@pytest.mark.parametrize("L", [4, 128, 132, 520, 1028, 4100])
@pytest.mark.parametrize("n,n_hot,share", [(2048, 1, 1.0), (2049, 1, 1.0), (2500, 3, 0.5), (5000, 12, 1.0), (8192, 1, 0.4), (8192, 8, 0.9)])
def test_small_pushes_with_hot_keys(n, n_hot, share, L):
    """Keys that are a large part of the call are shared by all blocks: integers exactly, and, with terms of very different
    size, the same bits again on a second store (whichever block finishes a key)."""
    K = 300
    rng = np.random.default_rng(n + L)
    keys = rng.integers(0, K, size=n)
    keys = np.where(rng.random(n) < share, 17 + 3 * rng.integers(0, n_hot, size=n), keys)
    upd = rng.integers(-4, 5, size=(n, L)).astype(np.float32)
    rough = (rng.normal(size=(n, L)) * 10.0 ** rng.choice([0, 5, 20], size=(n, 1))).astype(np.float32)
    (g, o), (h, _) = (make_pair(K, L, 3, max_batch_keys=n) for _ in range(2))
    rows = rng.integers(-100, 100, size=(K, L)).astype(np.float32)
    o.set_rows(np.arange(K), rows)
    for s in (g, h):
        s.set_all_rows(torch.from_numpy(rows))
        s.push(dev(keys), dev(upd))
    o.push(keys, upd)
    compare_state(g, o, exact_rows=True, what="hot keys")
    for s in (g, h):
        s.push(dev(keys), dev(rough))
        s.push(dev(keys[::-1].copy()), dev(upd))
        s.sync()
    assert torch.equal(g.export()[0], h.export()[0])


@pytest.mark.parametrize("mode,L,n,words", [("mf", 8, 4000, 1), ("mf", 260, 1500, 2), ("kge", 24, 700, 1), ("kge", 600, 500, 2),
                                            ("rescal", 16, 400, 1), ("sgns", 24, 500, 2), ("sgns", 300, 400, 1)])
def test_small_steps_with_hot_keys(mode, L, n, words):
    """Batches whose cells share a column, whose triples share a relation and few entities, of one or two words."""
    rng = np.random.default_rng(n)
    K, on_gpu, on_cpu = small_step(mode, 400 if mode == "mf" else words, words, L, n, rng)
    rows = np.abs(rng.normal(0.2, 0.05, size=(K, L))).astype(np.float32) * (0.1 if mode in ("mf", "sgns") else 1)
    g, o = make_pair(K, L, rows=rows, max_batch_keys=8192)
    on_gpu(g)
    on_cpu(o)
    g.sync()
    compare_state(g, o, what="hot keys in a small step")
    assert close(float(g.loss.cpu()[0]), o.loss[0])


def test_small_push_with_more_keys_in_one_bucket_than_its_table_holds():
    """Keys whose hash puts them all into the same block: the table overflows and warps compare for themselves."""
    K, L, n = 2_000_000, 4, 8000
    k = np.arange(K, dtype=np.uint64)
    h = ((k * 0x9E3779B1) & 0xFFFFFFFF) >> 16
    keys = k[h < 0x10000 // 400].astype(np.int64)[:n - 500]        # the lowest 1/400 of the hash range: one block of 295
    assert len(keys) > 3000
    g, o = make_pair(K, L, 1, max_batch_keys=n)
    rng = np.random.default_rng(5)
    keys = np.concatenate([keys, keys[rng.integers(0, len(keys), size=500)]])
    rng.shuffle(keys)
    upd = rng.integers(-4, 5, size=(len(keys), L)).astype(np.float32)
    g.push(dev(keys), dev(upd))
    o.push(keys, upd)
    g.sync()
    compare_state(g, o, exact_rows=True, what="overflowing bucket")


@pytest.mark.parametrize("n,dim,n_neg", [(1, 1, 1), (40, 7, 3), (64, 100, 10), (300, 12, 20), (20, 132, 4), (9, 1000, 29)])
def test_small_complex_steps(n, dim, n_neg):
    cfg = W.scaled(W.KGE_TINY, entities=300, dim=dim, n_neg=n_neg, batch=n, n_triples=4 * n)
    rows = W.kge_init_rows(cfg, 0, cfg.num_keys, "cpu")
    rows[:, 2 * dim:] = rows[:, :2 * dim].square() + 0.01           # accumulators some way into training
    g, o = make_pair(cfg.num_keys, cfg.row_len, 2, rows=rows, max_batch_keys=(3 + n_neg) * n)
    for b in range(3):
        s, r, ob, ne, ns = W.kge_triples(cfg, b * n, n, "cpu")
        args = (cfg.rel_key_base, dim, cfg.lr, cfg.eps)
        ps.ps_step_kge(g.h, s.cuda(), r.cuda(), ob.cuda(), ne.cuda(), ns.cuda(), n_neg, *args, g.loss)
        o.step_kge(s, r, ob, ne, ns, *args)
    g.sync()
    compare_state(g, o, what="small complex steps")
    assert close(float(g.loss.cpu()[0]), o.loss[0])
    ne[0, 0] = cfg.entities                                         # out of range: a no-op, loss included
    before = float(g.loss.cpu()[0])
    ps.ps_step_kge(g.h, s.cuda(), r.cuda(), ob.cuda(), ne.cuda(), ns.cuda(), n_neg, *args, g.loss)
    assert g.sync(check=False) == ps.PS_ERR_KEY_RANGE
    compare_state(g, o, what="small complex step with a bad index")
    assert float(g.loss.cpu()[0]) == before


@pytest.mark.parametrize("n,dim,n_neg", [(1, 129, 2), (74, 256, 4), (75, 257, 10), (148, 515, 3), (149, 512, 10), (33, 1028, 9),
                                         (700, 514, 10), (2, 130, 11), (50, 385, 20), (80, 260, 21), (160, 131, 29), (400, 258, 20)])
def test_wide_complex_steps(n, dim, n_neg):
    """Even dimensions: rows kept in shared memory.  Odd ones without a sort: streamed as finished rows, in clusters of four, two and one
    block per data point, stretches that do and do not divide among them and among the jobs of a pass, parts that start off a
    16-byte boundary, negatives shared by the halves of a block.  (Streamed gradients and rows updated in place: test_gpu_resident.)"""
    test_small_complex_steps(n, dim, n_neg)


@pytest.mark.parametrize("n,dim,n_neg", [(200, 66, 10), (41, 100, 5), (300, 128, 10), (300, 250, 10), (120, 1000, 10), (45, 1001, 29), (3, 4000, 20)])
def test_complex_steps_of_several_stretches_per_block(n, dim, n_neg):
    """Reductions whose blocks of all stretches are resident at once: one to 48 occurrences of a bucket, one to 16 stretches."""
    test_small_complex_steps(n, dim, n_neg)


@pytest.mark.parametrize("n", [1, 13, 2559, 2560, 2561, 4095, 4096, 4097])
@pytest.mark.parametrize("L", [200, 512, 700, 4100])
def test_small_pushes_around_the_limits_of_the_buckets(n, L):
    rng = np.random.default_rng(n + L)
    g, o = make_pair(n + 50, L, rows=rng.integers(-4, 5, size=(n + 50, L)).astype(np.float32), max_batch_keys=n)
    for share in (0.0, 0.5):
        keys = np.where(rng.random(n) < share, rng.integers(0, 9, size=n), rng.integers(0, n + 50, size=n))
        upd = rng.integers(-4, 5, size=(n, L)).astype(np.float32)
        g.push(dev(keys), dev(upd))
        o.push(keys, upd)
    g.sync()
    compare_state(g, o, exact_rows=True, what="pushes around the limits of the buckets")


@pytest.mark.parametrize("N,L,counts", [(8, 128, (1, 7, 600, 2047, 2048, 2049)), (1500, 4, (5, 700, 2048, 2500, 4000)),
                                        (3, 256, (2048, 1, 2049, 1025)), (8, 64, (1151, 1152, 1153))])
def test_localize_around_the_limit_of_the_single_launch(N, L, counts):
    K = 30_000
    g, o = make_pair(K, L, N, 2 * -(-K // N) + 4200, max_batch_keys=4000)
    rng = np.random.default_rng(N)
    for it, m in enumerate(counts * 2):
        w = int(rng.integers(0, N))
        keys = (rng.zipf(1.2, size=m) - 1) % K if it % 2 else rng.integers(0, K, size=m)
        g.localize(w, dev(keys))
        o.localize(w, keys)
        g.sync()
        compare_state(g, o, exact_rows=True, what=f"localize of {m}")
        upd = rng.integers(-2, 3, size=(m, L)).astype(np.float32)
        g.push(dev(keys), dev(upd))
        o.push(keys, upd)
    g.localize(0, dev(np.array([3, K])))
    assert g.sync(check=False) == ps.PS_ERR_KEY_RANGE
    compare_state(g, o, exact_rows=True, what="bad key")


@pytest.mark.parametrize("n", [600, 3_000])
def test_requested_counts_a_localize_that_finds_no_room(n):
    """On either side of the limit of the single launch."""
    K = 8_000
    g, _ = make_pair(K, 8, 2, K // 2 + 100, max_batch_keys=4096)
    g.localize(0, dev(np.arange(K - n, K)))
    assert g.sync(check=False) == ps.PS_ERR_CAPACITY
    g.localize(0, dev(np.arange(K - 50, K + 50) % K))
    g.sync()
    assert ps.ps_localize_stats(g.h) == {"requested": n + 100, "moved": 50, "already_local": 50, "moved_again": 0, "deferred": 0}


@pytest.mark.parametrize("n", [8_193, 16_384, 32_767, 32_768, 32_769, 303_104, 303_105, 606_300])
@pytest.mark.parametrize("K", [200, 70_000])
def test_sorted_pushes_around_the_limits_of_the_sorts(n, K):
    """The sort in one cluster, the cooperative one with a short tile per block and with longer ones: sizes around the
    changes, keys of one and of three digits, a key that is a third of the batch and runs of equal keys."""
    L = 4
    g, o = make_pair(K, L, 3, max_batch_keys=n)
    rng = np.random.default_rng(n + K)
    keys = rng.integers(0, K, size=n)
    keys[rng.random(n) < 0.33] = K // 3
    keys[n // 2:n // 2 + 3000] = K - 1
    upd = rng.normal(size=(n, L)).astype(np.float32)
    rows = torch.from_numpy(o.rows.copy())
    out = []
    for _ in range(2):                                              # the order of a key's terms is that of the call: same bits again
        g.set_all_rows(rows)
        g.push(dev(keys), dev(upd))
        g.sync()
        out.append(g.export(table=False)[0])
    assert torch.equal(out[0], out[1])
    o.push(keys, upd)
    compare_state(g, o, what=f"push of {n}")


@pytest.mark.parametrize("n", [300, 1_000, 2_500, 14_500, 29_000])
@pytest.mark.parametrize("pipelined", [False, True])
def test_skip_gram_reduction_at_every_tile_length(n, pipelined):
    """12,300 to 1.2M key occurrences: tiles of 8, 16, 32, 64 and 128 sorted positions, words that fill thousands of them and
    words that occur once; a batch that ends inside a tile and, clipped windows, with "no key" marks."""
    cfg = W.scaled(W.SGNS_TINY, vocab=20_000, n_tokens=n, dim=8, batch=n)
    rows = torch.from_numpy(np.random.default_rng(n).normal(0, 0.1, size=(cfg.num_keys, cfg.dim)).astype(np.float32))
    tokens, negs = W.sgns_tokens(cfg, 0, n, "cpu"), W.sgns_negatives(cfg, 0, n, "cpu")
    g, o = make_pair(cfg.num_keys, cfg.dim, rows=rows, max_batch_keys=n * (1 + 2 * cfg.window * (1 + cfg.n_neg)))
    ps.ps_set_pipelining(g.h, pipelined)
    ps.ps_step_sgns(g.h, tokens.cuda(), 0, n, cfg.window, negs.cuda(), cfg.n_neg, cfg.out_key_base, cfg.lr, g.loss)
    o.step_sgns(tokens, 0, n, cfg.window, negs, cfg.n_neg, cfg.out_key_base, cfg.lr)
    g.sync()
    compare_state(g, o, what=f"skip-gram, {n} centers")
    assert close(float(g.loss.cpu()[0]), o.loss[0])


@pytest.mark.parametrize("d,n_neg,batch,ents,rels", [(4, 0, 3_000, 500, 1), (28, 10, 700, 3_000, 300), (64, 3, 900, 500, 5),
                                                     (68, 10, 650, 800, 60), (128, 29, 200, 900, 2)])
def test_rescal_steps_with_a_sort(d, n_neg, batch, ents, rels):
    """Runs of relations from one data point to all 3,000 of the batch (pieces of four and of eight, chunks of every
    length), dimensions on both sides of the points kernel's two forms."""
    from tests.test_gpu_rescal import rescal_run
    rescal_run(d, n_neg, batch, ents, rels, steps=2, single_step=True, G=0.3)


@pytest.mark.parametrize("lr,eps", [(float("nan"), 1e-8), (float("inf"), 1e-8), (0.1, -1e-3), (0.1, 0.05)])
@pytest.mark.parametrize("mode,n", [("kge", 40), ("kge", 700), ("rescal", 40), ("rescal", 700)])
def test_adagrad_with_unusual_rates(mode, n, lr, eps):
    """Learning rates that are not finite, an eps that is negative or not small against the accumulators' roots:
    without and with a sort, keys that occur once, a few times and hundreds of times."""
    E, R, n_neg, L = 1_500, 3, 10, 48
    d = L // 4 if mode == "kge" else L // 2
    rng = np.random.default_rng(n)
    rows = np.abs(rng.normal(0, 0.4, size=(E + R * (d if mode == "rescal" else 1), L))).astype(np.float32) + 0.05
    g, o = make_pair(len(rows), L, rows=rows, max_batch_keys=(3 + n_neg + d) * n)
    s, t, ne = (((rng.zipf(1.3, size=z) - 1) % E).astype(np.uint32) for z in (n, n, (n, n_neg)))
    r, ns = rng.integers(0, R, size=n).astype(np.uint32), rng.integers(0, 2, size=(n, n_neg)).astype(np.uint8)
    step = ps.ps_step_kge if mode == "kge" else ps.ps_step_rescal
    step(g.h, *(dev(x, torch.int32) for x in (s, r, t, ne)), dev(ns), n_neg, E, d, lr, eps, g.loss)
    getattr(o, "step_" + mode)(s, r, t, ne, ns, E, d, lr, eps)
    g.sync()
    got = g.export(table=False)[0].numpy()
    assert (np.isfinite(got) == np.isfinite(o.rows)).all()
    assert (np.isnan(got) == np.isnan(o.rows)).mean() > 0.999       # (inf - inf: which of the two a sum of either sign becomes)
    ok = np.isfinite(got)
    assert close(got[ok], o.rows[ok]).all()


@pytest.mark.parametrize("batch", [512, 8192])
def test_losses_of_overlapped_host_steps_reach_pinned_and_pageable_words(batch):
    """Steps without and with a sort, each with a loss word of its own, every other one in pageable memory (a copy there, a
    kernel's store to pinned memory): all equal to what the device-batch calls accumulate."""
    cfg = W.scaled(W.MF_TINY, rows=3000, cols=400, rank=12, n_cells=6 * batch, batch=batch, lr=0.0005)
    rows = W.mf_init_rows(cfg, 0, cfg.num_keys, "cpu")
    i, j, v = W.mf_cells(cfg, W.mf_planted(cfg, "cpu"), 0, cfg.n_cells, "cpu")
    pinned = [t.pin_memory() for t in (i, j, v)]
    a, _ = make_pair(cfg.num_keys, cfg.rank, rows=rows, max_batch_keys=2 * batch)
    g, _ = make_pair(cfg.num_keys, cfg.rank, rows=rows, max_batch_keys=2 * batch)
    ps.ps_set_pipelining(g.h, True)
    ps.ps_set_host_overlap(g.h, True)
    words = [torch.zeros(1, dtype=torch.float64) for _ in range(cfg.n_batches)]
    words = [w.pin_memory() if b % 2 else w for b, w in enumerate(words)]
    want = []
    for b in range(cfg.n_batches):
        sl = slice(b * batch, (b + 1) * batch)
        ps.ps_step_mf(a.h, i[sl].cuda(), j[sl].cuda(), v[sl].cuda(), cfg.col_key_base, cfg.lr, cfg.lam, a.loss)
        a.sync()
        want.append(float(a.loss.cpu()[0]))
        ps.ps_step_mf_host(g.h, *(t[sl] for t in pinned), cfg.col_key_base, cfg.lr, cfg.lam, g.loss, words[b])
    g.sync()
    assert [float(w[0]) for w in words] == want


def small_step(mode, E, R, L, n, rng):
    """(number of keys, step(store) on the GPU, the same on the oracle) of a small step with random indexes."""
    d, q = {"kge": L // 4, "rescal": L // 2}.get(mode, L), 2
    u32 = lambda a: a.astype(np.uint32)
    if mode == "sgns":
        tok, neg = u32(rng.integers(0, E, size=n + 4)), u32(rng.integers(0, E, size=(n * 4, q)))
        a = [dev(tok, torch.int32), dev(neg, torch.int32)]
        return (2 * E, lambda g: ps.ps_step_sgns(g.h, a[0], 2, n, 2, a[1], q, E, 0.01, g.loss),
                lambda o: o.step_sgns(tok, 2, n, 2, neg, q, E, 0.01))
    i, j = u32(rng.integers(0, E, size=n)), u32(rng.integers(0, R, size=n))
    if mode == "mf":
        v = rng.normal(size=n).astype(np.float32)
        a = [dev(i, torch.int32), dev(j, torch.int32), dev(v)]
        return (E + R, lambda g: ps.ps_step_mf(g.h, *a, E, 0.01, 0.05, g.loss), lambda o: o.step_mf(i, j, v, E, 0.01, 0.05))
    t, ne = u32(rng.integers(0, E, size=n)), u32(rng.integers(0, E, size=(n, q)))
    ns = rng.integers(0, 2, size=(n, q)).astype(np.uint8)
    a = [dev(x, torch.int32) for x in (i, j, t, ne)] + [dev(ns)]
    step = ps.ps_step_kge if mode == "kge" else ps.ps_step_rescal
    return (E + R * (d if mode == "rescal" else 1), lambda g: step(g.h, *a, q, E, d, 0.1, 1e-8, g.loss),
            lambda o: getattr(o, "step_" + mode)(i, j, t, ne, ns, E, d, 0.1, 1e-8))


@pytest.mark.parametrize("L,mode", [(12, "mf"), (260, "mf"), (16, "kge"), (24, "sgns"), (300, "sgns"), (16, "rescal")])
def test_small_calls_back_to_back(L, mode):
    """Kernels of small calls are set up while the ones before them still run and write: relocation, step, push and pull over
    the same few keys, with nothing waited for, against the same calls waited for one by one (bit for bit) and the oracle."""
    rng = np.random.default_rng(L)
    steps = [small_step(mode, 60, 10, L, 40, rng) for _ in range(60)]
    K = steps[0][0]
    rows = np.abs(rng.normal(0.2, 0.1, size=(K, L))).astype(np.float32)
    calls = []
    for _, on_gpu, on_cpu in steps:
        keys, upd = rng.integers(0, K, size=50), np.abs(rng.normal(0, 0.01, size=(50, L))).astype(np.float32)
        calls.append((int(rng.integers(0, 3)), on_gpu, on_cpu, keys, upd, dev(keys), dev(upd)))
    (g, o), (h, _) = (make_pair(K, L, 3, K, rows=rows, max_batch_keys=4096) for _ in range(2))
    torch.cuda.synchronize()
    pulled = []
    for w, on_gpu, _, _, _, keys, upd in calls:
        g.localize(w, keys)
        on_gpu(g)
        g.push(keys, upd)
        pulled.append(g.pull(keys))
    g.sync()
    for (w, on_gpu, on_cpu, keys, upd, dk, du), got in zip(calls, pulled):
        for call in (lambda: h.localize(w, dk), lambda: on_gpu(h), lambda: h.push(dk, du)):
            call()
            h.sync()
        assert torch.equal(h.pull(dk), got)
        o.localize(w, keys)
        if got is pulled[0]:                # (the oracle's rows drift from the GPU's roundings over the later steps)
            on_cpu(o)
            o.push(keys, upd)
            assert close(got.cpu().numpy(), o.pull(keys)).all()
    for x, y in zip(g.export(), h.export()):
        assert torch.equal(x, y)
    assert torch.equal(g.loss, h.loss)
    o.set_rows(np.arange(K), g.export()[0].numpy())
    compare_state(g, o, exact_rows=True, what="tables and free lists")


@pytest.mark.parametrize("L", [4, 128, 260, 520])
@pytest.mark.parametrize("counts", [(8, 9, 16, 17, 32, 33), (9,) * 40, (33, 9, 64, 17, 9, 100, 12, 31, 40) * 3, (500, 9, 9, 300, 20)])
def test_small_pushes_with_several_long_keys_per_block(counts, L):
    """Keys of 4, 8 and 16 warps, several in one bucket of the call: sums exact on integers, and the same bits every time."""
    rng = np.random.default_rng(len(counts) + L)
    K = 3_000
    keys = rng.permutation(np.concatenate([np.repeat(rng.choice(K, len(counts), replace=False), counts), rng.integers(0, K, size=20)]))
    g, o = make_pair(K, L, rows=rng.integers(-50, 50, size=(K, L)).astype(np.float32))
    upd = rng.integers(-9, 9, size=(len(keys), L)).astype(np.float32)
    g.push(dev(keys), dev(upd))
    o.push(keys, upd)
    compare_state(g, o, exact_rows=True, what="integers")
    upd = rng.normal(size=(len(keys), L)).astype(np.float32)
    seen = []
    for _ in range(3):
        g.set_all_rows(torch.from_numpy(o.rows.copy()))
        g.push(dev(keys), dev(upd))
        seen.append(g.export(table=False)[0])
    o.push(keys, upd)
    compare_state(g, o, what="normal updates")
    assert torch.equal(seen[0], seen[1]) and torch.equal(seen[0], seen[2])


@pytest.mark.parametrize("L,counts", [(516, (3, 700, 1_500)), (1024, (2_048, 2_047)), (4100, (1, 40, 511, 512)), (448, (2_048, 2_049)),
                                      (452, (2_029, 2_030)), (1024, (1_600, 1_601)), (1028, (1_601, 2_040, 2_041))])
def test_localize_of_wide_rows_around_the_limit_of_the_single_launch(L, counts):
    """Rows that several warps move, a part each; both sides of each limit of the single launch: 1,600 keys, 3.5 MB and 8 MB of rows."""
    K, N = 2_500, 4
    g, o = make_pair(K, L, N, K, max_batch_keys=2_500)
    rng = np.random.default_rng(L)
    for it, m in enumerate(counts):
        keys = rng.integers(0, K, size=m)
        g.localize(it % N, dev(keys))
        o.localize(it % N, keys)
        g.sync()
        compare_state(g, o, exact_rows=True, what=f"localize of {m}")
