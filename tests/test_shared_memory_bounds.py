"""What a chain needs of a CTA's shared memory decides which chains are accepted, and which ladders
are resident at once: neither may shrink (host code, on the CPU; residency on the GPU)."""
import subprocess

import numpy as np
import pytest

from native_build import compile_host
from oracle import Oracle
from paper_1004_0023_gb300 import pt
from test_gpu_units import _problem


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
