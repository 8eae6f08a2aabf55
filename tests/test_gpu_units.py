"""The update units' edges against the oracle, bit for bit: the table-index bytes at the
largest Lmax of each form, copies that do not fill a unit, sites without and with many
neighbours, and every unit width. Tolerance zero, as in the other parity tests."""
import os

import numpy as np
import pytest

from oracle import Oracle
from paper_1004_0023_gb300 import instances
from paper_1004_0023_gb300 import pt

pytestmark = pytest.mark.gpu

THREADS = os.cpu_count() or 1


@pytest.fixture(scope="module", autouse=True)
def _lib(libpt):
    return libpt


def _problem(n, degree, P, R, lmax, seed):
    """Random graph of at most `degree` neighbours a site (site 0 has none); couplings as large
    as |h| + sum |J| = lmax allows at one site of each sign."""
    rng = np.random.default_rng(seed)
    deg = [0] * n
    ei, ej = [], []
    a, b = np.triu_indices(n, 1)
    for k in rng.permutation(a.size).tolist():
        i, j = int(a[k]), int(b[k])
        if i > 0 and deg[i] < degree and deg[j] < degree:
            deg[i] += 1
            deg[j] += 1
            ei.append(i)
            ej.append(j)
    top = max(1, (lmax - 1) // max(degree, 1))
    J = rng.integers(1, top + 1, len(ei)) * rng.choice([-1, 1], len(ei))
    load = np.zeros(n, np.int64)
    np.add.at(load, ei, np.abs(J))
    np.add.at(load, ej, np.abs(J))
    h = np.asarray([rng.integers(-1, 2) if load[i] < lmax else 0 for i in range(n)])
    h[0], h[1] = lmax, -(lmax - load[1])
    beta = 8.0 / lmax  # thresholds spread over the whole table
    T = np.linspace(1.0, 2.0, R) * P / beta / 4
    gamma = np.linspace(0.4, 1.5, R) * T
    return instances.Problem(n, np.asarray(ei, np.int32), np.asarray(ej, np.int32), J.astype(np.int32),
                             h.astype(np.int32), P, T, gamma, 0xABC0 + seed)


CASES = [
    # one copy a thread (path 1, and path 9 for a short ladder)
    (9, 4, 2, 3, 9, {}), (9, 4, 6, 3, 41, {}), (12, 5, 10, 4, 42, {}), (20, 9, 18, 3, 60, {}), (34, 32, 34, 2, 127, {}),
    (12, 3, 32, 4, 7, {}), (16, 7, 24, 5, 127, {}), (3, 0, 64, 3, 5, {}), (10, 3, 300, 2, 6, {}),
    # path 1, a word of four copies a thread
    (9, 4, 2, 3, 9, dict(kernel_path=1, threads_per_block=96)), (11, 5, 14, 3, 41, dict(kernel_path=1, threads_per_block=64)),
    (20, 9, 12, 3, 42, dict(kernel_path=1, threads_per_block=96)), (34, 32, 34, 2, 127, dict(kernel_path=1, threads_per_block=128)),
    (16, 3, 16, 3, 31, dict(kernel_path=1, threads_per_block=32)),
    # paths 2, 3, 5, 6, 8: largest narrow and smallest wide index, both neighbour classes
    *[(14, d, 16, 4, lmax, dict(kernel_path=path)) for path in (2, 3, 5, 6, 8) for d, lmax in
      ((3, 41), (3, 42), (7, 41), (7, 127))],
    # path 4: nibble words (P % 32 == 0, Lmax <= 31) and one bit a copy
    *[(14, d, P, 3, lmax, dict(kernel_path=4)) for d in (3, 6, 7) for P, lmax in
      ((32, 31), (96, 13), (32, 32), (40, 31), (64, 42))],
    # path 7: units of one, two and four words
    *[(40, d, P, 3, lmax, dict(kernel_path=7, group_threads=32)) for d, lmax in ((3, 41), (7, 41), (3, 42), (7, 42))
      for P in (8, 16, 48, 128)],
]


@pytest.mark.parametrize("k", range(len(CASES)))
def test_unit_edges_match_the_oracle(k):
    n, degree, P, R, lmax, kw = CASES[k]
    prob = _problem(n, degree, P, R, lmax, k)
    g, o = pt.PT.from_problem(prob, **kw), Oracle.from_problem(prob, threads=THREADS)
    assert g.info.lmax == lmax
    moved = 0
    for sweeps in (1, 1, 2, 30):
        g.run(sweeps, 1)
        o.run(sweeps, 1)
        assert np.array_equal(g.read_state(), o.read_state()), (CASES[k], sweeps)
        og, oo = g.obs(), o.obs()
        for key in oo:
            assert np.array_equal(np.asarray(og[key]), np.asarray(oo[key])), (CASES[k], sweeps, key)
        moved = int(np.sum(og["flip_acc"]))
    assert moved > 0


BATCH = [(n, d, P, R, lmax) for n, d, lmax in ((24, 3, 31), (24, 3, 32), (30, 6, 31), (30, 7, 41), (20, 7, 42), (130, 3, 8))
         for P, R in ((8, 5), (24, 3), (32, 4), (64, 3), (96, 6), (128, 2))] + [(700, 3, 128, 9, 9), (1000, 6, 64, 20, 30)]


@pytest.mark.parametrize("cluster", [1, 2, 0])
def test_batched_chain_forms_match_the_oracle(cluster):
    """Every form of a batched chain (int8 rows in units of 1, 2 and 4 words, nibble and bit
    words), resident and streamed, over two runs; cluster 0 is timed at create and then reused
    from the cache, which has to bring its own groups to the device."""
    probs = [_problem(*c, 100 + k) for k, c in enumerate(BATCH)]
    for k, p in enumerate(probs):
        p.n_sweeps, p.sweeps_per_swap = 4 + k % 3, 1 + k % 2
    batches = [pt.Batch(probs, cluster_size=cluster)]
    if cluster == 0:
        assert batches[0].info().tuned_layouts >= 2
        batches.append(pt.Batch(probs))
        assert batches[1].info().tuned_layouts == 0
    for b in batches:
        orcs = [Oracle.from_problem(p, threads=THREADS) for p in probs]
        for run in range(2):
            b.run()
            for k, (p, o) in enumerate(zip(probs, orcs)):
                o.run(p.n_sweeps, p.sweeps_per_swap)
                assert np.array_equal(b.read_state(k), o.read_state()), (BATCH[k], run)
                og, oo = b.obs(k), o.obs()
                for key in oo:
                    assert np.array_equal(np.asarray(og[key]), np.asarray(oo[key])), (BATCH[k], run, key)


@pytest.mark.parametrize("n,degree,P,R,lmax,pieces", [
    (512, 3, 64, 6, 13, True), (512, 1, 64, 4, 5, False), (500, 7, 64, 5, 41, False), (512, 7, 64, 4, 42, False),
    (420, 3, 72, 5, 31, False), (300, 5, 120, 3, 60, False),
])
def test_chains_whose_random_words_do_not_fit_whole_match_the_oracle(n, degree, P, R, lmax, pieces):
    """Automatic plans of chains too large for two sweeps of produced words: path 8 makes them in
    pieces of a sweep. `pieces`: it is the fastest there by a quarter, so it has to be the plan."""
    prob = _problem(n, degree, P, R, lmax, n + P)
    g, o = pt.PT.from_problem(prob), Oracle.from_problem(prob, threads=THREADS)
    assert g.info.kernel_path == 8 or not pieces
    for sweeps, sps in ((1, 1), (2, 1), (7, 0), (12, 3)):
        g.run(sweeps, sps)
        o.run(sweeps, sps)
        assert np.array_equal(g.read_state(), o.read_state())
    og, oo = g.obs(), o.obs()
    for k in oo:
        assert np.array_equal(np.asarray(og[k]), np.asarray(oo[k])), k
    g.close()


@pytest.mark.parametrize("kw", [dict(), *[dict(kernel_path=k) for k in (1, 2, 3, 4, 5, 8, 9)],
                                dict(kernel_path=9, threads_per_block=96, producer_threads=32),
                                dict(P=1, kernel_path=1), dict(P=1, kernel_path=10)])
def test_back_to_back_launches_match_the_oracle(kw):
    """Sweep, swap and run launches of two contexts enqueued in turn without a wait between them:
    a launch's set-up may overlap the one before, its sweeps may not."""
    kw = dict(kw)
    P = kw.pop("P", 0)
    probs = [_problem(16, 3, P or 32, 6, 9, 7), _problem(40, 5, P or 48, 9, 30, 8)]
    if P == 1:  # classical chains have no transverse field
        for p in probs:
            p.gamma = np.zeros_like(p.gamma)
    gs = [pt.PT.from_problem(p, **kw) for p in probs]
    os_ = [Oracle.from_problem(p, threads=THREADS) for p in probs]
    x = [np.where(np.random.default_rng(k).random(o.read_state().shape) < 0.5, 1, -1).astype(np.int8)
         for k, o in enumerate(os_)]
    for round_ in range(3):
        for step in range(12):
            for c in gs + os_:
                c.sweep(1 + step % 3)
                c.swap()
                if step % 4 == 3:
                    c.run(4, 2)
        for g, o in zip(gs, os_):
            assert np.array_equal(g.read_state(), o.read_state()), round_
        if round_ == 0:
            for k in range(2):
                gs[k].write_state(x[k])
                os_[k].write_state(x[k])
    for g, o in zip(gs, os_):
        og, oo = g.obs(), o.obs()
        for k in oo:
            assert np.array_equal(np.asarray(og[k]), np.asarray(oo[k])), k
        g.close()


def test_an_unequal_backlog_on_wide_clusters_matches_the_oracle():
    """Nine requests admitted together, the longest by far the largest: clusters wider than one for
    each member, which the shorter ones take in turn."""
    probs = [_problem(120, 7, 64, 32, 30, 3)] + [_problem(12 + k, 3, 16 + 8 * (k % 3), 4 + k, 9, k) for k in range(8)]
    for k, p in enumerate(probs):
        p.n_sweeps, p.sweeps_per_swap = 30 if k == 0 else 12, 1 + k % 3
    srv = pt.Server(arena_bytes=1 << 28)
    ids = [srv.submit(p) for p in probs]
    done = set()
    while len(done) < len(ids):
        done |= set(srv.step())
    for rid, p in zip(ids, probs):
        state, obs = srv.result(rid)
        o = Oracle.from_problem(p, threads=THREADS)
        o.run(p.n_sweeps, p.sweeps_per_swap)
        assert np.array_equal(state, o.read_state())
        want = o.obs()
        for k in want:
            assert np.array_equal(np.asarray(obs[k]), np.asarray(want[k])), k
    srv.close()


# both neighbour classes, narrow and wide index, copies that don't fill 16; the last four with
# records that don't fit beside the words (two pieces) and with whole sweeps' words that don't
PIECES = [(60, 3, 64, 6, 13), (60, 7, 64, 5, 41), (60, 7, 64, 4, 42), (60, 3, 40, 4, 127)]
PIECES = [(*c, k) for c in PIECES for k in (2, 3, 5, 8)] + [
    (500, 7, 64, 4, 41, 2), (500, 7, 64, 4, 60, 2), (512, 3, 64, 5, 13, 4), (512, 3, 64, 5, 42, 8)]


@pytest.mark.parametrize("case", PIECES)
def test_random_words_in_pieces_match_the_oracle(case):
    """Path 8 with its words in a given number of pieces, whatever plan would be the fastest."""
    prob = _problem(*case[:5], 300 + case[5])
    g, o = pt.PT.from_problem(prob, kernel_path=8, test_pieces=case[5]), Oracle.from_problem(prob, threads=THREADS)
    assert g.info.kernel_path == 8 and 2 <= g.info.pieces <= case[5]
    for sweeps, sps in ((1, 1), (2, 1), (7, 0), (12, 3), (1, 0)):
        g.run(sweeps, sps)
        o.run(sweeps, sps)
        assert np.array_equal(g.read_state(), o.read_state()), (sweeps, sps)
    og, oo = g.obs(), o.obs()
    for k in oo:
        assert np.array_equal(np.asarray(og[k]), np.asarray(oo[k])), k
    g.close()


@pytest.mark.parametrize("pieces", [2, 3, 8])
def test_partner_that_never_publishes_times_out_with_words_in_pieces(pieces):
    """The sweeping CTA gives up with sweeps left and skips to the sweep's last barrier; the word CTA
    meets it at its next piece's, learns of it there and leaves with it."""
    prob = _problem(60, 3, 64, 6, 13, 9)
    g = pt.PT.from_problem(prob, kernel_path=8, test_pieces=pieces, wait_timeout_ms=200, test_withhold_rung=3,
                           swap_mode=1)
    assert g.info.pieces >= 2
    g.run(4, 1)
    with pytest.raises(pt.PTError) as e:
        g.sync()
    assert e.value.code == pt.PT_ETIMEDOUT
    g.close()
    h, o = pt.PT.from_problem(prob), Oracle.from_problem(prob, threads=THREADS)
    h.run(20, 1)
    o.run(20, 1)
    assert np.array_equal(h.read_state(), o.read_state())


@pytest.mark.parametrize("n,degree,P,lmax,threads", [
    (400, 3, 32, 31, 0), (400, 3, 32, 13, 96), (250, 3, 96, 31, 0), (700, 6, 32, 31, 0), (300, 6, 96, 30, 0),
    (800, 7, 32, 31, 0), (300, 7, 128, 29, 512), (120, 2, 192, 5, 0),
])
def test_nibble_words_on_large_levels_match_the_oracle(n, degree, P, lmax, threads):
    """Path 4 on levels of at least 224 one-bit units, which take 16 copies a unit: the largest Lmax
    of the form, every number of neighbour slots, rows of several words."""
    prob = _problem(n, degree, P, 3, lmax, n + P)
    g, o = pt.PT.from_problem(prob, kernel_path=4, threads_per_block=threads), Oracle.from_problem(prob, threads=THREADS)
    assert 2 * n * (P // 8) // g.info.n_levels >= 224
    for sweeps, sps in ((1, 1), (2, 1), (6, 0), (10, 3)):
        g.run(sweeps, sps)
        o.run(sweeps, sps)
        assert np.array_equal(g.read_state(), o.read_state()), (sweeps, sps)
    og, oo = g.obs(), o.obs()
    for k in oo:
        assert np.array_equal(np.asarray(og[k]), np.asarray(oo[k])), k
