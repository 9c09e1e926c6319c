"""The rules that choose a form of the moment loop's step (CPU only)."""
import os
import shutil
import subprocess
import time

import pytest

import kpm_workloads as W
import paper_2104_13218_gb300 as kpm
from paper_2104_13218_gb300 import _lib

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def route(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    _lib.lib()  # builds libkpm.so if needed
    libdir = os.path.join(ROOT, "paper_2104_13218_gb300", "_build")
    exe = str(tmp_path_factory.mktemp("route") / "route_dump")
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_2104_13218_gb300", "csrc"), "-I" + cuda_inc,
                    os.path.join(HERE, "host", "route_dump.cpp"), "-o", exe, "-L" + libdir, "-lkpm",
                    "-Wl,-rpath," + libdir], check=True)

    def run(model, n_up, R, precision="fp64", K=200):
        bonds = [f"{i} {j} {J!r}" for i, j, J in zip(model.bi, model.bj, map(float, model.J))]
        text = " ".join(map(str, [model.n_sites, R, K, int(precision == "fp32"), len(n_up), *n_up,
                                  len(bonds), *bonds]))
        out = subprocess.run([exe], input=text, check=True, capture_output=True, text=True).stdout.split()
        assert out[0] == "0"
        return {k: int(v) for k, v in zip(out[1::2], out[2::2])}

    return run


# A step in fixed point rounds a component by 0.29/U in the root mean square, one with
# FP64 vectors by 2^-53.8 .. 2^-54.05 (both in units of 1/sqrt(D)): no model may be given a
# unit at which the first is larger.  One and two groups, and couplings of their own,
# from few to the most bonds, with and without the small-sector kernel.
@pytest.mark.parametrize("n,k", [(12, 6), (18, 9), (23, 11)])
def test_fixed_point_rounds_no_more_than_fp64(route, n, k):
    pairs = [(i, j) for j in range(n) for i in range(j)]
    seen = set()
    for count in (1, 12, 20, 40, 44, 51, 52, 66, 84, 101, 102, 120, 153, 253):
        if count > len(pairs):
            continue
        for kind in ("one", "two", "own"):
            J = {"one": lambda b: 1.0, "two": lambda b: 1.0 + (b % 2), "own": lambda b: 1.0 + 0.01 * b}[kind]
            model = W._model(kind, n, [(i, j, J(b)) for b, (i, j) in enumerate(pairs[:count])])
            r = route(model, [k], 16)
            if r["small"] or r["fixed"]:
                assert 0.29 / r["unit"] <= 2 ** -54.05, (kind, count, r)
                seen.add(kind)
    assert seen == {"one", "two", "own"}


# Lists padded for the fixed-point kernel may not fit where those of the FP64 kernel do: a run
# that had lists keeps them, for every number of vectors.
@pytest.mark.parametrize("model", [W.ring(18), W.j1j2_chain(18, 1.0, 0.4), W.ladder(18), W.sawtooth(18, -1.0, 0.4),
                                   W.j1j2_square(4, 5, 1.0, 0.5)], ids=lambda m: m.name)
def test_fixed_point_keeps_the_lists(route, model):
    for R in list(range(3, 34)) + [48, 64, 65, 100, 128, 129]:
        r = route(model, [model.n_sites // 2], R)
        assert r["stride"] > 0 or r["fp64_stride"] == 0, (R, r)


# Small sectors run in one launch where that is the faster form: not when a few vectors of
# a large sector would leave most of the chip idle, nor when the kernels that spread a step over the
# chip fill it as well.  (the clear cases of the measurements: the other form at least 20% slower)
@pytest.mark.parametrize("model,n_up,R,one_launch", [
    (W.j1j2_chain(16, 1.0, 0.4), [8], 1, 0), (W.j1j2_chain(16, 1.0, 0.4), [8], 4, 0),
    (W.j1j2_chain(16, 1.0, 0.4), [8], 16, 0), (W.random_bonds(16, 32, 3, 0.2, 1.5), [8], 1, 0),
    (W.random_bonds(16, 32, 3, 0.2, 1.5), [8], 16, 0), (W.j1j2_chain(15, 1.0, 0.4), [7], 8, 0),
    (W.j1j2_chain(15, 1.0, 0.4), [7], 4, 0),
    (W.random_bonds(15, 30, 3, 0.2, 1.5), [8, 9, 10], 4, 0), (W.ladder(16), [8, 9, 10, 11, 12, 13, 14, 15, 16], 8, 0),
    (W.ladder(14), [7], 1, 1), (W.ladder(14), [7, 8, 9, 10, 11, 12, 13, 14], 25, 1), (W.ring(10), [-1], 20, 1),
    (W.ring(12), [6], 1, 1), (W.ring(16), [-1], 100, 1), (W.ladder(16), [8, 9, 10, 11, 12, 13, 14, 15, 16], 1, 1)])
def test_small_sectors_rule(route, model, n_up, R, one_launch):
    assert route(model, n_up, R)["small"] == one_launch


# The bounds need the plan of the states alone: with the plans of a whole space's sectors on top
# their size query (and call) took five times as long, longer than for a sector of it.
def test_bounds_prepare_no_more_than_the_plan():
    model = W.ring(16)

    def shortest(n_up):
        t = []
        for _ in range(60):
            t0 = time.perf_counter()
            kpm.bounds_workspace_size(model, n_up)
            t.append(time.perf_counter() - t0)
        return min(t)

    assert shortest([-1]) < shortest([8])
