"""The box-tree search (k_nn.cu) at the edges of its leaves (8 points), query groups (4 and 16), nodes
(256), super nodes (8192) and of the rule that picks the group, against exhaustive search.

Coordinates are multiples of 1/64, so every squared distance is exact in FP32 and in the oracle's
FP64, ties are everywhere, and the indices must match exactly (lowest index on ties): no
tolerance.  Zero grids and a zero learning rate keep the moving points where they are; two steps
run, the first without and the second with the previous neighbours."""
import numpy as np
import pytest

from oracle import pdg_oracle as O

pytestmark = pytest.mark.gpu


def lattice(seed, n, spread):
    r = np.random.Generator(np.random.PCG64(seed))
    return (np.round(r.uniform(-spread, spread, (n, 3)) * 64) / 64).astype(np.float32)


@pytest.mark.parametrize("V,N,M,spread", [
    (1, 1, 1, 1.0), (7, 9, 8, 0.5), (31, 33, 32, 1.4), (255, 257, 256, 1.0), (257, 5, 1, 0.2),
    (8193, 3, 8191, 1.4), (1000, 9000, 9001, 1.0), (300, 70, 400, 40.0)])  # the last: far outside the domain
def test_indices_match_exhaustive_search(V, N, M, spread):
    from paper_2509_18097_gb300 import binding as B

    X, S, T = lattice(1, V, spread), lattice(2, N, spread), lattice(3, M, spread)
    cfg = B.pdg_config_default(res=(2, 4), lr0=0.0)
    ctx = B.pdg_create(cfg, X, np.zeros((0, 2), np.int32), S, max_pts=max(N, M))
    try:
        B.pdg_begin_frame(ctx, T)
        for _ in range(2):
            B.pdg_step(ctx, 1)
            fwd = B.pdg_read(ctx, B.BUF_NN_FWD, 0, np.empty(V + N, np.int32))
            rev = B.pdg_read(ctx, B.BUF_NN_REV, 0, np.empty((2, M), np.int32))
            for got, q, b in ((fwd[:V], X, T), (fwd[V:], S, T), (rev[0], T, X), (rev[1], T, S)):
                assert np.array_equal(got, O.nn_bruteforce(q, b)[0])
    finally:
        B.pdg_destroy(ctx)
