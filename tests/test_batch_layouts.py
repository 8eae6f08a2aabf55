"""Batched layouts with streamed chains: which CTAs stream and which keep their chains, and the
sequence of their tasks (host code, on the CPU), and the bits of the requests that have both (GPU)."""
import os
import subprocess
import time

import numpy as np
import pytest

from native_build import compile_host
from oracle import Oracle
from paper_1004_0023_gb300 import pt
from test_gpu_units import _problem

THREADS = os.cpu_count() or 1

# n, degree, P, R, Lmax, cluster: the last CTA of the cluster holds no more chains than groups while
# the others stream (byte units of one and four words, wide index, nibble words) ...
MIXED = [(200, 6, 64, 33, 9, 2), (1024, 3, 128, 10, 60, 4), (1024, 3, 96, 33, 9, 4), (444, 3, 120, 31, 9, 5),
         (444, 3, 120, 31, 9, 8)]
# ... and every CTA streams (bit words among them)
STREAMED = [(294, 6, 128, 45, 20, 1), (900, 7, 40, 35, 60, 2)]


@pytest.fixture(scope="module")
def native(libpt, tmp_path_factory):
    """native(name): the host program tests/native/<name>.cu, compiled once."""
    out_dir = tmp_path_factory.mktemp("native")
    built = {}

    def program(name):
        if name not in built:
            built[name] = compile_host(name, out_dir)
        return built[name]

    return program


@pytest.fixture(scope="module")
def layouts(native):
    exe = native("batch_layouts")

    def run(problems):
        text = []
        for p in problems:
            text.append("%d %d %d %d" % (p.n, len(p.ei), p.P, p.R))
            text += ["%d %d %d" % edge for edge in zip(p.ei, p.ej, p.J)]
            text.append(" ".join(str(int(x)) for x in p.h))
        r = subprocess.run([exe], input="\n".join(text) + "\n0 0 0 0\n", capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        out = []
        for line in r.stdout.splitlines():
            head, ctas = line.split("|")
            P, R, lmax, K, form, group, n_groups, resident, buffers, nbytes = map(int, head.split())
            c = list(map(int, ctas.split()))
            out.append(dict(P=P, R=R, lmax=lmax, K=K, form=form, group=group, n_groups=n_groups, resident=resident,
                            buffers=buffers, bytes=nbytes,
                            ctas=[dict(count=c[x], keep=c[x + 1], in_place=c[x + 2]) for x in range(0, 3 * K, 3)]))
        return out

    return run


def test_a_cta_that_keeps_its_chains_does_not_stream_them(layouts):
    """A kept chain has one buffer for the run and no other group waits for it, so no copy of it may
    be in flight between sweeps; and every CTA has the buffers its chains take."""
    rng = np.random.default_rng(3)
    cases = [c[:5] for c in MIXED + STREAMED]
    for _ in range(60):
        n, d, P = int(rng.integers(32, 1025)), int(rng.integers(3, 8)), 8 * int(rng.integers(1, 17))
        cases.append((n, d, P, int(rng.integers(2, 129)), int(rng.choice([9, 30, 41, 60]))))
    found = layouts([_problem(*c, k) for k, c in enumerate(cases)])
    assert len(found) == 16 * len(cases)
    both = 0
    for lay in found:
        if lay["bytes"] < 0:
            continue
        assert sum(c["count"] for c in lay["ctas"]) == lay["R"]
        for c in lay["ctas"]:
            assert c["in_place"] or not c["keep"], lay
            assert not c["in_place"] or c["count"] <= lay["buffers"], lay
        live = [c for c in lay["ctas"] if c["count"]]
        both += any(c["in_place"] for c in live) and not all(c["in_place"] for c in live)
    assert both > 10
    for k, c in enumerate(MIXED + STREAMED):
        lay = found[16 * k + c[5] - 1]
        assert lay["bytes"] > 0 and not lay["resident"], c
        kept = [x["in_place"] for x in lay["ctas"] if x["count"]]
        assert any(kept) == (c in MIXED) and not all(kept), c


@pytest.mark.parametrize("chains,first", [
    (1024, 0), (1024, 2 ** 21 - 3), (1024, 2 ** 22 - 3), (1024, 2 ** 30 - 40), (32, 2 ** 26 - 40), (32, 2 ** 30 - 40),
    (17, 2 ** 31 // 17 - 5), (17, 2 ** 30 - 40),
])
def test_tasks_of_the_longest_runs_stay_in_range(native, chains, first):
    """2^30 sweeps of 1024 chains: the task number passes 2^31, 2^32 and ends at 2^40."""
    groups = 16
    r = subprocess.run([native("batch_tasks"), str(chains), str(2 ** 30), str(first), "60000", str(groups)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) == min(60000, (2 ** 30 + 1 - first) * chains - groups)


@pytest.mark.gpu
@pytest.mark.parametrize("case", MIXED + STREAMED)
def test_streamed_and_kept_chains_of_one_request_match_the_oracle(libpt, case):
    prob = _problem(*case[:5], 40 + case[0])
    prob.n_sweeps, prob.sweeps_per_swap = 6, 2
    b = pt.Batch([prob], cluster_size=case[5])
    o = Oracle.from_problem(prob, threads=THREADS)
    for run in range(2):
        b.run()
        o.run(prob.n_sweeps, prob.sweeps_per_swap)
        assert np.array_equal(b.read_state(0), o.read_state()), run
        og, oo = b.obs(0), o.obs()
        for key in oo:
            assert np.array_equal(np.asarray(og[key]), np.asarray(oo[key])), (run, key)


@pytest.mark.gpu
@pytest.mark.parametrize("case", [(16, 3, 32, 6, 9, 1), (24, 3, 32, 40, 9, 2), (24, 3, 32, 5, 9, 4), MIXED[0], MIXED[1],
                                  STREAMED[1]])
def test_batched_waits_end_at_the_given_limit(libpt, case):
    """The chain on rung 2 never publishes: its partner's wait ends after wait_timeout_ms and the
    call returns PT_ETIMEDOUT, with chains kept, taken as tasks and streamed; a new batch then runs."""
    prob = _problem(*case[:5], 60 + case[0])
    prob.n_sweeps, prob.sweeps_per_swap = 8, 1
    b = pt.Batch([prob, prob], cluster_size=case[5], wait_timeout_ms=150, test_withhold_rung=2)
    start = time.monotonic()
    b.run()
    with pytest.raises(pt.PTError) as e:
        b.sync()
    assert e.value.code == pt.PT_ETIMEDOUT
    assert time.monotonic() - start < 4.0
    with pytest.raises(pt.PTError):  # sticky
        b.run()
    b.close()
    b = pt.Batch([prob], cluster_size=case[5])
    b.run()
    o = Oracle.from_problem(prob, threads=THREADS)
    o.run(prob.n_sweeps, prob.sweeps_per_swap)
    assert np.array_equal(b.read_state(0), o.read_state())
