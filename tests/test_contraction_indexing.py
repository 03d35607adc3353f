"""Index safety of the contraction streams (D2Q9, D2Q16, D3Q27), checked on the CPU.

The step kernels restate here in float32 / float64 and Python integers: the rule that lets a
node take the contraction (every departure floor is -1 or 0), the staged window it then reads
(two nodes either side), the places of the slots for every tile shape, the ring of the
non-local terms at periodic and zero-gradient edges, and the shared memory of a block."""
import numpy as np
import pytest

HALO, NB, SPLIT = 2, 128, 12
AUX, KQ, KEEP, SL = 4, 5, 36, 32
MAX_SMEM = 227 * 1024            # a block's shared memory on this part
TILES = [(tx, NB // tx, False) for tx in (1, 2, 4, 8, 16, 32, 64, 128)] + [
    (tx, 64 // tx, False) for tx in (16, 32, 64)] + [(tx, SPLIT // tx, True) for tx in (1, 2, 4, 6, 12)]
GAUGES = [0.0, 1e-30, 0.05, 0.5, 0.9999999, 1.0, 1.7, 3.0, 1e4, 1e38, np.inf, np.nan]
C16 = np.sqrt(3 - np.sqrt(6.0)), np.sqrt(3 + np.sqrt(6.0))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("comps", [(-1.0, 0.0, 1.0), (-C16[1], -C16[0], C16[0], C16[1])])
def test_window_holds_every_stencil_of_the_contraction(dtype, comps):
    rng = np.random.default_rng(5)
    us = [x for g in GAUGES for x in (g, -g)] + list(rng.uniform(-2.5, 2.5, 200))
    taken = 0
    with np.errstate(all="ignore"):
        for s in GAUGES + list(rng.uniform(0.01, 2.0, 60)):
            for u in us:
                for dt in (0.1, 0.5, 1.0):
                    d = [-(dtype(s) * dtype(c) + dtype(u)) * dtype(dt) for c in comps]
                    f = np.floor(d)
                    if not all(x == 0 or x == -1 for x in f):      # (NaN: not taken)
                        continue
                    taken += 1
                    assert all(np.isfinite(d)) and max(np.abs(d)) <= 1
                    for x in f:
                        # five columns from -2; a floor of 0 reads the last four, -1 the first
                        assert -HALO <= x - 1 and x + 2 <= HALO
                        assert (1 if x == 0 else 0) == int(x) - 1 + HALO
    assert taken > 1000


@pytest.mark.parametrize("tx,ty,split", TILES)
def test_slots_of_a_tile(tx, ty, split):
    wt, n = tx + 2 * HALO, (tx + 2 * HALO) * (ty + 2 * HALO)
    k = np.arange(n)
    cv = ((k.astype(np.float32) + np.float32(0.5)) * (np.float32(1) / np.float32(wt))).astype(int)
    assert (cv == k // wt).all()                                # the quotient by a reciprocal
    rw = tx + 2
    r = np.arange(rw * (ty + 2))
    j = ((r.astype(np.float32) + np.float32(0.5)) * (np.float32(1) / np.float32(rw))).astype(int)
    assert (j == r // rw).all()
    for ly in range(ty):
        for lx in range(tx):
            own = (ly + HALO) * wt + lx + HALO
            assert 0 <= own - HALO * (wt + 1) and own + HALO * (wt + 1) < n
            c0 = (ly + 1) * rw + lx + 1                           # ring: stress and flux, one node around
            assert 0 <= c0 - rw - 1 and c0 + rw + 1 < rw * (ty + 2)


@pytest.mark.parametrize("tx,ty,split", TILES)
@pytest.mark.parametrize("n", [1, 2, 3, 7, 16, 129, 300])
def test_ring_nodes_at_the_edges_of_the_grid(tx, ty, split, n):
    """A zero-gradient edge moves a ring node onto the grid; its 3 x 3 slots are staged."""
    for t in (tx, ty):
        for x0 in range(0, n, t):
            for i in range(t + 2):
                for clamp in (False, True):
                    m = min(max(x0 + i - 1, 0), n - 1) if clamp else x0 + i - 1
                    c = m - (x0 - HALO)
                    assert 1 <= c <= t + 2


@pytest.mark.parametrize("size", [4, 8])
def test_shared_memory_of_a_block(size):
    for tx, ty, split in TILES:
        slots, stride9, stride16 = (tx + 4) * (ty + 4), (20, 19)[size == 8], (36, 33)[size == 8]
        own = SPLIT * (SL + 9 * 18) if split else NB * KEEP
        assert (slots * (AUX + stride9) + (tx + 2) * (ty + 2) * KQ + own) * size + 2048 <= MAX_SMEM
        if not split:
            assert NB * (10 * 8 + 36 * size) + slots * stride16 * size + 2048 <= MAX_SMEM
    # D3Q27: 8 x 4 x 4 nodes, 12 x 8 staged per plane, planes padded by eight slots
    plane = 12 * 8 + 8
    own = [(z + 2) * plane + (y + 2) * 12 + x + 2 for z in range(4) for y in range(4) for x in range(8)]
    reach = 2 * plane + 2 * 12 + 2
    assert min(own) - reach >= 0 and max(own) + reach < 8 * plane
    assert max(k + 8 * (k // 96) for k in range(12 * 8 * 8)) < 8 * plane
    assert 8 * plane * (30, 27)[size == 8] * size + (24 * NB * 4 if size == 4 else 0) + 2048 <= MAX_SMEM
