"""The bit-sliced classification (tc_sliced.cuh) compiled for the host, all
threads of a block phase by phase, against the oracle (no GPU needed)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import tcurve_inputs as ti
from triangulations import apex_triangulation, greedy_triangulation, hub_triangulation

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = "/usr/local/cuda"


@pytest.fixture(scope="module")
def sliced_exe(tmp_path_factory):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    csrc = os.path.join(ROOT, "paper_2604_09221_gb300", "csrc")
    out = {}
    for groups in (2, 4, "blocks"):
        exe = tmp_path_factory.mktemp("sliced") / f"run{groups}"
        name = "run_block_sliced.cpp" if groups == "blocks" else "run_sliced_sweep.cpp"
        cmd = ["g++", "-std=c++17", "-O1", "-w", f"-DTC_SL_GROUPS={groups}", f"-I{csrc}",
               f"-I{os.path.join(HERE, 'host')}", f"-I{os.path.join(ROOT, 'oracle')}",
               f"-I{CUDA}/include", "-o", str(exe), os.path.join(HERE, "host", name),
               "-x", "c", os.path.join(ROOT, "oracle", "tcurve_oracle.c"), "-x", "none",
               f"-L{CUDA}/lib64", f"-Wl,-rpath,{CUDA}/lib64", "-lcudart", "-lpthread"]
        subprocess.run(cmd, check=True, capture_output=True)
        out[groups] = exe
    return out


@pytest.mark.parametrize("d", list(range(1, 17)))
def test_sliced_sweep_on_the_host(sliced_exe, tmp_path, d):
    """Random and special sign vectors on the standard, (d >= 3) a regular and
    (d >= 2) the fan triangulation, whose origin has more earlier neighbours
    than a vertex's row of label planes holds takes for: one- and two-byte
    labels, both back ends, blocks of 64 and 128 sign vectors, every area of
    exactly the kernels' size."""
    cases = [("standard", ti.standard_triangulation(d))]
    if d >= 3:
        cases.append(("regular", ti.regular_triangulation(d, seed=300 + d)))
    if d >= 2:
        cases.append(("fan", ti.fan_triangulation(d)))
    for name, edges in cases:
        np.savetxt(tmp_path / "tri.txt", edges, fmt="%d")
        for groups in (2, 4):
            exe = sliced_exe[groups]
            out = subprocess.run([str(exe), str(d), str(tmp_path / "tri.txt"), "3"],
                                 capture_output=True, text=True)
            assert out.returncode == 0, (name, groups, out.stdout + out.stderr)


@pytest.mark.parametrize("d", [4, 5, 6, 7, 8, 9])
def test_block_sweep_on_the_host(sliced_exe, tmp_path, d):
    """The bit-sliced block sweep: the halves of 128 high parts (the first,
    the last and random ones) and every middle-row pattern of each, per mask
    map, against the oracle's histogram of the same masks; standard, regular,
    fan and (d = 8) the printed triangulations.  The middle phase takes every
    high part but those of the fan triangulation at d = 9 (too many open
    components: the kernel takes those mask by mask)."""
    cases = [("standard", ti.standard_triangulation(d)), ("regular", ti.regular_triangulation(d, seed=d)),
             ("fan", ti.fan_triangulation(d))]
    if d == 8:
        cases += [(n, np.loadtxt(os.path.join(HERE, "golden", f"fig2_{n}.edges"), dtype=np.int32, comments="#"))
                  for n in ("rank016", "rank015")]
    for k, (name, edges) in enumerate(cases):
        np.savetxt(tmp_path / "tri.txt", edges, fmt="%d")
        maps = [("plain", d + 1), ("flip", d), ("reduced", d - 1), ("orbits", d + 1)]
        for mode, ib in maps if name == "regular" else maps[:1]:
            if ib < 5:
                continue
            out = subprocess.run([str(sliced_exe["blocks"]), str(d), str(tmp_path / "tri.txt"), mode, str(k)],
                                 capture_output=True, text=True)
            assert out.returncode == 0, (name, mode, out.stdout + out.stderr)
            taken = int(out.stdout.split("middle phase=")[1].split()[0])
            assert taken == (0 if (name, d) == ("fan", 9) else 128), out.stdout


def _block_sweep(exe, tmp_path, d, edges, mode, seed=1):
    """Run the block sweep's host emulation; it agrees with the oracle.
    Returns how many of the 128 high parts the middle phase took."""
    np.savetxt(tmp_path / "tri.txt", edges, fmt="%d")
    out = subprocess.run([str(exe), str(d), str(tmp_path / "tri.txt"), mode, str(seed)],
                         capture_output=True, text=True)
    assert out.returncode == 0, (mode, out.stdout + out.stderr)
    return int(out.stdout.split("middle phase=")[1].split()[0])


MAPS = {"plain": 1, "flip": 0, "reduced": -1, "orbits": 1}  # middle-row bits less d


def _maps(d, every):
    return [m for m, b in MAPS.items() if d + b >= 5 and (every or m == "plain")]


@pytest.mark.parametrize("d,k", [(d, k) for d in range(4, 10) for k in range(1, d) if np.gcd(d, k) == 1])
def test_block_sweep_keeps_vertex_0_beside_the_middle_row(sliced_exe, tmp_path, d, k):
    """An edge (0, d)-(k, 0): the first vertex of the sweep is a neighbour of
    the middle row."""
    for mode in _maps(d, every=k == {5: 2, 6: 1, 7: 3, 8: 3, 9: 2}.get(d)):
        taken = _block_sweep(sliced_exe["blocks"], tmp_path, d, apex_triangulation(d, k), mode)
        assert taken == (0 if d >= 8 and k in (1, d - 1) else 128)


@pytest.mark.parametrize("d,n", [(6, 7), (6, 8), (7, 8), (8, 8), (8, 9), (9, 8), (9, 9)])
def test_block_sweep_takes_fans_of_any_length(sliced_exe, tmp_path, d, n):
    """The origin has 31, 35 or 39 earlier neighbours and the middle phase
    takes every high part."""
    for mode in _maps(d, every=n == 8):
        assert _block_sweep(sliced_exe["blocks"], tmp_path, d, hub_triangulation(d, n), mode) == 128


@pytest.mark.parametrize("d", [5, 6, 7, 8, 9])
def test_block_sweep_on_random_triangulations(sliced_exe, tmp_path, d):
    """Twenty triangulations with edges of any length, each in one mask map."""
    maps = _maps(d, every=True)
    for seed in range(20):
        _block_sweep(sliced_exe["blocks"], tmp_path, d, greedy_triangulation(d, seed), maps[seed % len(maps)])


@pytest.fixture(scope="module")
def open_exe(sliced_exe, tmp_path_factory):
    csrc = os.path.join(ROOT, "paper_2604_09221_gb300", "csrc")
    exe = tmp_path_factory.mktemp("open") / "run"
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", f"-I{csrc}", f"-I{os.path.join(ROOT, 'oracle')}",
                    f"-I{CUDA}/include", "-o", str(exe), os.path.join(HERE, "host", "run_open_components.cpp"),
                    "-x", "c", os.path.join(ROOT, "oracle", "tcurve_oracle.c"), "-x", "none",
                    f"-L{CUDA}/lib64", f"-Wl,-rpath,{CUDA}/lib64", "-lcudart", "-lpthread"],
                   check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("d", [5, 6, 7, 8, 9])
def test_the_host_knows_what_the_middle_phase_holds(open_exe, sliced_exe, tmp_path, d):
    """A triangulation's components next to the middle row, counted when it is
    loaded: the same for every sign vector, and within the middle phase's limit
    exactly if it takes the high parts."""
    held = set()
    for edges in ([ti.standard_triangulation(d), ti.fan_triangulation(d), apex_triangulation(d, 1)]
                  + [greedy_triangulation(d, seed) for seed in range(8)]):
        np.savetxt(tmp_path / "tri.txt", edges, fmt="%d")
        out = subprocess.run([str(open_exe), str(d), str(tmp_path / "tri.txt"), "300"],
                             capture_output=True, text=True)
        assert out.returncode == 0, out.stderr
        n, most = map(int, out.stdout.split())
        mode = "reduced" if d > 5 else "plain"
        assert (_block_sweep(sliced_exe["blocks"], tmp_path, d, edges, mode) == 128) == (n <= most)
        held.add(n <= most)
    assert held == {True, False}


@pytest.mark.parametrize("d", [13, 14])
def test_wide_blocks_on_the_host(tmp_path, d):
    """Blocks of 192 sign vectors: standard, fan and a random triangulation."""
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    csrc, exe = os.path.join(ROOT, "paper_2604_09221_gb300", "csrc"), tmp_path / "run"
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-DTC_SL_GROUPS=6", f"-I{csrc}",
                    f"-I{os.path.join(ROOT, 'oracle')}", f"-I{CUDA}/include", "-o", str(exe),
                    os.path.join(HERE, "host", "run_sliced_sweep.cpp"),
                    "-x", "c", os.path.join(ROOT, "oracle", "tcurve_oracle.c"), "-x", "none",
                    f"-L{CUDA}/lib64", f"-Wl,-rpath,{CUDA}/lib64", "-lcudart", "-lpthread"],
                   check=True, capture_output=True)
    for edges in (ti.standard_triangulation(d), ti.fan_triangulation(d), greedy_triangulation(d, 3)):
        np.savetxt(tmp_path / "tri.txt", edges, fmt="%d")
        out = subprocess.run([str(exe), str(d), str(tmp_path / "tri.txt"), "2"], capture_output=True, text=True)
        assert out.returncode == 0, out.stdout + out.stderr
