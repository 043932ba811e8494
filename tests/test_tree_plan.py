"""The cluster kernel's launch shapes (host code, on the CPU): the device's largest
cluster and SM count bound them."""

import os
import shutil
import subprocess

import pytest

from tests.test_abi import ROOT, _cuda_lib_dir

SMEM_SM, SMEM_BLOCK = 233472, 232448


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    """plans([(B, R, V, logit_bytes, sms, max_cluster), ...]) -> [(ncw, C, stages, smem, ok,
    fits), ...]; further entries force the shape."""
    from paper_2505_12398_gb300.build import build
    cxx, cudadir = shutil.which("g++"), _cuda_lib_dir()
    if not cxx or not cudadir:
        pytest.skip("no C++ compiler or CUDA runtime library")
    libdir = os.path.dirname(build())
    exe = str(tmp_path_factory.mktemp("plan") / "plan")
    r = subprocess.run([cxx, "-std=c++17", "-I", os.path.join(os.path.dirname(cudadir), "include"),
                        "-I", "/usr/local/cuda/include",
                        "-I", os.path.join(ROOT, "paper_2505_12398_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "c_abi", "plan.cc"), "-o", exe, "-L", libdir,
                        "-ltv", f"-Wl,-rpath,{libdir}", f"-Wl,-rpath-link,{cudadir}",
                        f"-Wl,-rpath,{cudadir}"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(cases):
        text = "".join("%d %d %d %d %d %d %d %d %d %d %d\n" %
                       (c[:5] + (SMEM_SM, SMEM_BLOCK, c[5]) + tuple(c[6:] or (0, 0, 0)))
                       for c in cases)
        r = subprocess.run([exe], input=text, capture_output=True, text=True, timeout=120)
        assert r.returncode == 0
        out = [tuple(int(x) for x in line.split()) for line in r.stdout.splitlines()]
        assert len(out) == len(cases)
        return out
    return run


BATCHES = (1, 4, 8, 9, 16, 17, 32, 33, 76, 77, 224, 225, 320, 512, 513, 4096)


@pytest.mark.parametrize("most", [16, 8, 4, 2, 1])
def test_clusters_the_device_can_hold(plans, most):
    """No plan asks for a larger cluster than the device holds, whether chosen or forced."""
    cases = [(B, R, V, lb, 152, most) + f for B in BATCHES for R in (2, 61, 121)
             for V in (1000, 32000, 128256, 262144) for lb in (2, 4)
             for f in ((), (8, 16, 0), (16, 8, 0))]
    got = plans(cases)
    assert all(p[1] <= most and p[4] for p in got)
    if most == 16:
        assert {p[1] for p in got} == {1, 2, 4, 8, 16}
        # few trees of long rows take whole SMs, many of short ones half of one each
        got = plans([(1, 61, 128256, 2, 152, 16), (32, 61, 128256, 2, 152, 16),
                     (1024, 61, 32000, 2, 152, 16)])
        assert [p[:2] for p in got] == [(16, 16), (8, 8), (8, 1)]


def test_batches_count_against_the_sms(plans):
    """Half the SMs: the shapes of twice the batch."""
    whole = plans([(2 * B, 61, 128256, 2, 152, 16) for B in BATCHES])
    half = plans([(B, 61, 128256, 2, 76, 16) for B in BATCHES])
    assert whole == half


def test_every_size_taken_has_a_plan(plans):
    """The largest trees and vocabularies the entry points accept: two ring stages at
    least, whatever the batch."""
    cases = []
    for R in (1, 2, 200, 500, 800, 1000, 1016, 1024):
        room = (SMEM_BLOCK - 64 - 97 * R) // 8 * 256     # the largest vocabulary accepted
        for V in [1, 1000, 262144] + [room * k // 64 for k in range(16, 65)]:
            cases += [(B, R, V, lb, 152, most) for B in BATCHES for lb in (2, 4)
                      for most in (16, 8)]
    got = plans(cases)
    assert all(p[5] for p in got)
    assert [c for c, p in zip(cases, got) if not p[4] or p[2] < 2] == []
