"""The three-pass 2-D transform of the fused kernels (csrc/fft3.cuh) on the host (CPU only): its source run
thread by thread against a direct DFT in double precision, and the shared-memory banks of its exchanges.
"""
import os
import pathlib
import shutil
import subprocess

import pytest

HERE = pathlib.Path(__file__).resolve().parent
CSRC = HERE.parent / "paper_2406_06640_gb300" / "csrc"
CUDA_INC = pathlib.Path(os.environ.get("CUDA_HOME", "/usr/local/cuda")) / "include"


@pytest.fixture(scope="module")
def emu(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx or not (CUDA_INC / "cuda_runtime.h").exists():
        pytest.skip("g++ and the CUDA headers are needed to compile the FFT source for the host")
    exe = tmp_path_factory.mktemp("fft3emu") / "fft3_host_emu"
    r = subprocess.run([cxx, "-std=c++20", "-O2", f"-I{CUDA_INC}", f"-I{CSRC}", str(HERE / "fft3_host_emu.cpp"),
                        "-o", str(exe), "-lpthread"], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    assert r.returncode == 0, r.stdout
    return exe


@pytest.mark.parametrize("M", [64, 128])
def test_source_matches_a_direct_dft(emu, M):
    r = subprocess.run([str(emu), str(M)], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
    _, fwd, _, rt, _, guard = r.stdout.split()
    # FP32 butterflies and twiddles: ~1e-7 relative per transform (log2(M^2) stages)
    assert float(fwd) < 5e-6 and float(rt) < 5e-6 and guard == "1", r.stdout


@pytest.mark.parametrize("M", [64, 128])
def test_exchanges_are_free_of_bank_conflicts(M):
    """8-byte accesses: the 16 lanes of a half warp in 16 different 8-byte banks; 16-byte accesses: the 8 lanes of
    a quarter warp in 8 different 16-byte banks, at even slots."""
    S, NT, TH = M // 64, M // 16, 4 * M
    L1 = TH + 2
    slots1, slots2 = set(), set()
    for tid0 in range(0, TH, 16):
        lanes = range(tid0, tid0 + 16)
        for s in range(S):
            for k2 in range(16):
                w = [t + k2 * L1 + s * 16 * L1 for t in lanes]
                assert len({x % 16 for x in w}) == 16
                slots1.update(w)
        for k1 in range(NT):
            for ka in range(4):
                w = [t % 16 + M * (4 * (t // 16 % 16) + 64 * (t // 256)) + 16 * k1 + M * ka for t in lanes]
                assert len({x % 16 for x in w}) == 16
                slots2.update(w)
        for s in range(S):
            for i in range(16):
                assert len({(t % M + M * (t // M) + M * (4 * i + 64 * s)) % 16 for t in lanes}) == 16
        for q in (0, 8):
            for ya in range(4):
                for t in range(0, NT, 2):
                    r = [(l // 256) * 16 * L1 + (l % 16) * L1 + (l // 16 % 16) * NT + ya * 16 * NT + t
                         for l in range(tid0 + q, tid0 + q + 8)]
                    assert all(x % 2 == 0 for x in r) and len({x // 2 % 8 for x in r}) == 8
                    assert set(r) <= slots1 or max(r) < 16 * S * L1
    assert len(slots1) == M * M and max(slots1) < 16 * S * L1 and slots2 == set(range(M * M))
