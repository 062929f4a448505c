"""The rule up to which a launch gives every particle three lanes follows the
device's number of multiprocessors: a small host program compiled from the
header that states it."""
import os
import shutil
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cuda_runtime.h>
#include <cmath>
#include "mp_internal.h"
#include "mp_sched.cuh"
int main()
{
    for (int warps : {12, 20})
        for (int sms : {1, 76, 132, 148, 152}) {
            const long long limit = 10LL * warps * sms;
            if (!mp::few_particles(1, warps, sms) || !mp::few_particles(limit, warps, sms) ||
                mp::few_particles(limit + 1, warps, sms)) {
                printf("%d warps, %d multiprocessors\n", warps, sms);
                return 1;
            }
        }
    return 0;
}
"""


def test_limit_follows_the_device():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "rule.cu"), os.path.join(d, "rule")
        with open(src, "w") as f:
            f.write(PROGRAM)
        subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                               "-I", os.path.join(ROOT, "include"),
                               "-I", os.path.join(ROOT, "paper_2302_13590_gb300", "csrc"), src, "-o", exe])
        r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
        assert r.returncode == 0, r.stdout + r.stderr
    for name in ("mp_fp64.cu", "mp_mixed.cu"):
        with open(os.path.join(ROOT, "paper_2302_13590_gb300", "csrc", name)) as f:
            assert "sm_count(&sms)" in f.read(), name
