"""What a chain needs of a CTA's shared memory decides which chains are accepted, and which ladders
are resident at once: neither may shrink (host code, on the CPU; residency on the GPU)."""
import subprocess

from native_build import compile_host


def test_no_layout_asks_for_more_than_its_data_and_800_bytes(libpt, tmp_path):
    r = subprocess.run([compile_host("layout_bounds", tmp_path)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout.split()[0]) > 10000
