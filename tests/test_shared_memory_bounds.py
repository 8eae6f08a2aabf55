"""What a chain needs of a CTA's shared memory decides which chains are accepted, and which ladders
are resident at once: neither may shrink (host code, on the CPU; residency on the GPU)."""
import subprocess

import numpy as np
import pytest

from native_build import compile_host
from oracle import Oracle
from paper_1004_0023_gb300 import pt
from test_gpu_units import _problem
from test_zz_no_alloc import _device_problem, _state_of


def test_no_layout_asks_for_more_than_its_data_and_800_bytes(libpt, tmp_path):
    r = subprocess.run([compile_host("layout_bounds", tmp_path)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout.split()[0]) > 10000


def test_chains_that_fit_one_cta_with_a_threshold_row_are_held_at_any_group_width(libpt, tmp_path):
    """Path 7 with a given width: every group has a threshold row of its own, so where the widest
    count of groups leaves no room for the chains, fewer groups hold them."""
    cases = []
    for P, R, lmax, dc in ((256, 2, 88, 8), (144, 1, 43, 4), (8, 16, 42, 4), (8, 40, 112, 8), (64, 5, 7, 4)):
        # the largest N whose chains fit beside one row and 400 bytes
        fixed = 4 * (3 * (2 * lmax + 1)) + 200 + R * 56 + 60 * 4 + 400
        n = (227 * 1024 - 1024 - fixed) // (P * R + (32 if dc == 4 else 48) + 8) - 1
        cases += ["%d %d %d %d %d 60 1 %d" % (n, P, R, lmax, dc, g) for g in (32, 64, 128, 256, 512)]
    r = subprocess.run([compile_host("resident_groups", tmp_path)], input="\n".join(cases), capture_output=True,
                       text=True)
    got = [tuple(map(int, x.split())) for x in r.stdout.splitlines()]
    assert r.returncode == 0 and len(got) == len(cases)
    for c, (groups, nbytes) in zip(cases, got):
        assert 1 <= groups <= 512 // int(c.split()[-1]) and nbytes <= 227 * 1024 - 1024, (c, groups, nbytes)
    assert any(groups < 512 // int(c.split()[-1]) for c, (groups, _) in zip(cases, got))


@pytest.mark.gpu
@pytest.mark.parametrize("n,P,R,lmax,group", [(1320, 8, 16, 42, 32), (509, 136, 3, 43, 64)])
def test_fewer_groups_than_the_cta_has_match_the_oracle(libpt, n, P, R, lmax, group):
    """Chains that fill the CTA, on path 7 with a given width."""
    prob = _problem(n, 3, P, R, lmax, n)
    g, o = pt.PT.from_problem(prob, kernel_path=7, cluster_size=1, group_threads=group), Oracle.from_problem(prob)
    for sweeps, sps in ((2, 1), (5, 2)):
        g.run(sweeps, sps)
        o.run(sweeps, sps)
        assert np.array_equal(g.read_state(), o.read_state())


# ladders of several CTAs an SM that the simplest kernel of the path holds at once: one copy a thread,
# the automatic plan's, held level-0 units, nibble words at the widest block, words from a second CTA,
# split chains
LADDERS = [
    (8, 3, 10, 700, dict(kernel_path=1)), (8, 3, 12, 700, dict()), (9, 5, 20, 800, dict(kernel_path=1)),
    (8, 3, 16, 700, dict(kernel_path=2, threads_per_block=128)), (8, 3, 16, 700, dict(kernel_path=3, threads_per_block=128)),
    (8, 3, 32, 250, dict(kernel_path=4, threads_per_block=512)), (8, 5, 16, 250, dict(kernel_path=4, threads_per_block=448)),
    (16, 3, 24, 700, dict(kernel_path=7, group_threads=512, cluster_size=4)),
    (8, 3, 16, 100, dict(kernel_path=8, threads_per_block=320)), (8, 3, 16, 250, dict(kernel_path=6, threads_per_block=160)),
]


@pytest.mark.gpu
@pytest.mark.parametrize("n,degree,P,R,kw", LADDERS)
def test_long_ladders_stay_resident(libpt, n, degree, P, R, kw):
    prob = _problem(n, degree, P, R, 9, n + R)
    g = pt.PT.from_problem(prob, swap_mode=1, **kw)
    assert g.info.cooperative == 1
    o = Oracle.from_problem(prob)
    for sweeps, sps in ((3, 1), (2, 0), (6, 2)):
        g.run(sweeps, sps)
        o.run(sweeps, sps)
        assert np.array_equal(g.read_state(), o.read_state())
    og, oo = g.obs(), o.obs()
    for k in oo:
        assert np.array_equal(np.asarray(og[k]), np.asarray(oo[k])), k


@pytest.mark.gpu
def test_long_ladders_stay_resident_on_callers_memory(libpt):
    torch = pytest.importorskip("torch")
    prob = _problem(8, 3, 32, 700, 9, 5)
    ref, o = pt.PT.from_problem(prob), Oracle.from_problem(prob)
    dp, bufs = _device_problem(torch, prob, ref, None)
    pt.run_noalloc(dp, 6, 2, 0, None)
    o.run(6, 2)
    got = _state_of(torch, bufs, prob)
    assert got["status"] == 0 and np.array_equal(got["state"], o.read_state())
