"""Calls whose scratch does not fit in its default form."""
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

import kpm_workloads as W
import paper_2104_13218_gb300 as kpm

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


# A device whose allocations fail above a limit (refused on the host, in the test program): the
# call is made with the kernels that need the least scratch.  FP32 runs on lists with matrix
# elements repeat the sums of the matrix-free ones; FP64 within the parity tests' 1e-10.
def test_failed_allocations(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    libdir = os.path.join(ROOT, "paper_2104_13218_gb300", "_build")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    exe = str(tmp_path / "alloc_limit")
    subprocess.run([cxx, "-O1", "-std=c++17", "-rdynamic", "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(cuda, "include"), os.path.join(HERE, "host", "alloc_limit.cpp"), "-o", exe,
                    "-L" + libdir, "-lkpm", "-L" + os.path.join(cuda, "lib64"), "-lcudart", "-ldl",
                    "-Wl,-rpath," + libdir, "-Wl,-rpath," + os.path.join(cuda, "lib64")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()
    assert len(out) >= 10
    for line in out:
        name, rc, rc_limit, diff = line.split()[:4]
        tol = 1e-5 if name in ("moments-0-12-1", "moments-0-16-1") else 1e-10
        # (grouped FP32 runs have no form with less scratch)
        if name == "gradient-outside":
            assert int(rc) == 0 and int(rc_limit) == 2, line
            continue
        if name == "moments-0-16-1":
            assert int(rc) == 0 and int(rc_limit) in (0, 2), line
            continue
        assert int(rc) == 0 and int(rc_limit) == 0 and float(diff) <= tol, line


# A caller's workspace that holds only that form, full of NaN patterns.
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("R", [4, 25, 33])
def test_moments_in_a_small_workspace(R, precision):
    for model, n_up in ((W.j1j2_chain(16, 1.0, 0.4), [8, 5]), (W.random_bonds(16, 37, 3, -0.7, 0.7), [8])):
        S = len(n_up)
        kw = dict(a=[16.0] * S, b=[0.0] * S, precision=precision, device=True)
        ref = kpm.moments(model, n_up, 12, R, 5, **kw)
        size = kpm.moments_workspace_size(model, n_up, 12, R, precision)
        lo, hi = 0, size  # the least size that is accepted
        while hi - lo > 4096:
            mid = (lo + hi) // 2 // 256 * 256
            ws = torch.full((max(mid, 256),), 0xFF, dtype=torch.uint8, device="cuda")
            try:
                got = kpm.moments(model, n_up, 12, R, 5, workspace=ws, **kw)
                hi = mid
            except kpm.KPMError as e:
                assert "KPM_ENOMEM" in str(e)
                lo = mid
                continue
            for q in ("mu", "mu_M", "mu_M2"):
                scale = ref[q].abs().clamp(min=1.0)
                assert ((got[q] - ref[q]).abs() / scale).max() <= (1e-10 if precision == "fp64" else 1e-5), (q, mid)
        if model.n_bonds == 37 and (R > 4 or precision == "fp64"):  # (FP32 rows of one lane have no lists)
            assert hi < 0.8 * size  # without the lists with matrix elements


# A caller's workspace without room for the FP64 sweep's checkpoints: enough for a run in fixed
# point, KPM_ENOMEM for one that leaves the range; the queried size serves both.
def test_gradient_in_a_small_workspace():
    model, n_up, K, R = W.j1j2_chain(14, 1.0, 0.4), [7], 200, 20
    cls = model.classes()
    g = {"mu": np.cos(1.0 + np.arange(K))[None]}
    size = kpm.moments_backward_workspace_size(model, n_up, K, R)
    small = size - 2 * 4 * 3432 * R * 8  # the pairs of every 32nd of 100 steps
    for bytes_, a, enough in ((small, 30.0, True), (small, 1.0, False), (size, 1.0, True)):
        args = (model, cls, 2, n_up, [a], [0.0], K, R, 5, g)
        ws = torch.full((bytes_ + 4096,), 0xFF, dtype=torch.uint8, device="cuda")
        if not enough:
            with pytest.raises(kpm.KPMError, match="KPM_ENOMEM"):
                kpm.moments_backward(*args, workspace=ws)
            continue
        got, ref = kpm.moments_backward(*args, workspace=ws), kpm.moments_backward(*args)
        assert np.array_equal(got, ref), (a, got, ref)


# What the library keeps between calls (up to 256 MB) can be had back, and it works on.
def test_kept_scratch_is_given_back():
    model, kw = W.ring(16), dict(a=[6.0], b=[-1.0], device=True)
    first = kpm.moments(model, [8], 20, 60, 5, **kw)["mu"]
    kpm.moments(W.ring(18), [9], 10, 100, 5, **kw)  # two vectors of 39 MB
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    kpm.release_scratch()
    assert torch.cuda.mem_get_info()[0] - before >= 64 << 20
    kpm.release_scratch()
    assert torch.equal(kpm.moments(model, [8], 20, 60, 5, **kw)["mu"], first)


# A problem whose default scratch exceeds the static array and whose least does not.
def test_static_scratch_takes_the_least_form():
    model, n_up, K, R = W.random_bonds(19, 38, 3, -0.7, 0.7), [9], 12, 10
    assert kpm.moments_workspace_size(model, n_up, K, R, "fp64") > kpm.lib().kpm_static_scratch_bytes()
    a, b, nu = np.array([16.0]), np.array([0.5]), np.array(n_up, dtype=np.int32)
    mu = torch.full((1, K), float("nan"), dtype=torch.float64, device="cuda")
    rc = kpm.lib().kpm_moments_static(kpm.CModel.of(model).ref, 1, nu.ctypes.data, a.ctypes.data, b.ctypes.data, K, R,
                                      5, 0, 0, mu.data_ptr(), None, None, torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    ref = kpm.moments(model, n_up, K, R, 5, a=a, b=b)["mu"]
    assert np.abs(mu.cpu().numpy() - ref).max() <= 1e-10
