"""The row gather's sub-walks (host logic, no GPU): tests/split_replay.cu cuts
every row's walk into 1, 2, 4 and 8 sub-walks with the library's split_walk,
replays them as the lanes of a row do and compares with direct sums over the
star in double (1e-12: a few hundred roundings of 1.1e-16 each)."""
import os
import re
import subprocess

import pytest

from tests.test_walk_encoder_cpu import CASES, ROOT, _nvcc, _write


@pytest.fixture(scope="module")
def replay(tmp_path_factory):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = tmp_path_factory.mktemp("split") / "split_replay"
    cmd = [nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
           os.path.join(ROOT, "tests", "split_replay.cu"), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return exe


@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_sub_walks_replay_the_star(replay, tmp_path, name, make):
    mesh, u = make()
    f = tmp_path / "mesh.bin"
    _write(f, mesh, u)
    r = subprocess.run([str(replay), str(f)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    stats = dict(re.findall(r"(\w+)=([0-9.eE+-]+)", r.stdout))
    assert int(stats["elements"]) == 4 * 4 * mesh.n_elems  # every star once per number of sub-walks
