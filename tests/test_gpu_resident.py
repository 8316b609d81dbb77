"""GPU parity of ComplEx on rows that stay in shared memory: chunks of 64 dimensions and their remainders, every alignment of a row's second
half, one to 32 rows per data point, clusters for few data points and for wide rows; both sides of the last sizes that fit a block, a
cluster of two and one of four, and the streamed kernel beyond them."""
import numpy as np
import pytest
import torch

import paper_2002_00655_b200 as ps
from tests.test_gpu_sorted import EPS, LR, ada_rows, check, check_no_op, on_gpu, triples
from tests.util import make_pair

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
