"""What a device is asked once (svh::AnswerPerDevice in csrc/sv_host.h), driven on the host with a fake of the runtime: an answer is kept, per device
and 0 included; a failed query is not, and clears its own error; a query that succeeds leaves an earlier error of the caller's alone."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include "sv_host.h"
static int device, cleared, asked;
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = device; return device < 0 ? cudaErrorUnknown : cudaSuccess; }
cudaError_t cudaGetLastError() { ++cleared; return cudaSuccess; }
}
#define EXPECT(x) if (!(x)) return printf("line %d: " #x "\n", __LINE__), 1
int main()
{
    static svh::AnswerPerDevice known;
    auto ask = [](int answer) { return known.get([=] { ++asked; return answer; }); };
    EXPECT(ask(-1) == 0 && asked == 1 && cleared == 1);   // a failure is no answer
    EXPECT(ask(33) == 33 && asked == 2 && cleared == 1);
    EXPECT(ask(7) == 33 && asked == 2);
    device = 1;
    EXPECT(ask(0) == 0 && asked == 3 && ask(5) == 0 && asked == 3 && cleared == 1);
    device = svh::kMaxDevices;
    EXPECT(ask(5) == 0 && asked == 3);
    device = 0;
    EXPECT(ask(5) == 33 && asked == 3 && cleared == 1);
    return 0;
}
"""


def test_answers_are_kept_and_failures_are_not(tmp_path):
    nvcc = next((c for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")) if c and os.path.exists(c)), None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    (tmp_path / "answers.cpp").write_text(DRIVER)
    exe = str(tmp_path / "answers")
    cuda = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2512_21911_b200", "csrc"), "-I", cuda,
                    str(tmp_path / "answers.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
