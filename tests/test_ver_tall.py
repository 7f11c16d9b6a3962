"""The voxel error rate's indexing: the division of voxel indices over its whole range (CPU), and
volumes of more than 2^23 rows (GPU), which an FP32 quotient cannot tell apart."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2211_03516_gb300", "csrc", "exact_div.cuh")

CHECK = r"""
#include "%s"
#include <stdio.h>
int main() {
    const uint32_t last = 2147483647u;
    uint64_t seed = 1, n = 0;
    auto rnd = [&] { seed = seed * 6364136223846793005ull + 1442695040888963407ull; return (uint32_t)(seed >> 33); };
    auto check = [&](uint32_t d) {
        const vamrt::ExactDiv q(d);
        auto one = [&](uint32_t i) {
            if (i > last) return true;
            ++n;
            if (q(i) == i / d) return true;
            printf("%%u / %%u = %%u, not %%u\n", i, d, i / d, q(i));
            return false;
        };
        // beside multiples of d: the first, the last, and some between
        for (int k = 0; k < 400; ++k) {
            const uint32_t most = last / d, c = k == 0 ? 0 : k == 1 ? most : k == 2 && most ? most - 1 : (uint32_t)(rnd() %% (most + 1ull));
            for (int e = -1; e <= 1; ++e)
                if (!one((uint32_t)((int64_t)c * d + e < 0 ? 0 : (int64_t)c * d + e))) return false;
        }
        return one(last);
    };
    for (uint32_t d = 1; d < 3000; ++d) if (!check(d)) return 1;
    for (int s = 0; s < 31; ++s)
        for (int e = -1; e <= 1; ++e) {
            const int64_t d = ((int64_t)1 << s) + e;
            if (d >= 1 && !check((uint32_t)d)) return 1;
        }
    if (!check(last)) return 1;
    for (int k = 0; k < 3000; ++k) if (!check(rnd() %% last + 1)) return 1;
    printf("%%llu\n", (unsigned long long)n);
    return 0;
}
"""


def test_exact_division(tmp_path):
    cc = shutil.which("g++") or shutil.which("c++")
    if cc is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(CHECK % HEADER)
    subprocess.run([cc, "-O2", "-std=c++17", str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 5_000_000


@pytest.mark.gpu
# one voxel per read; 16 bytes of FP32; 16 bytes of BF16.  FP32 quotients with one correction lose
# 905102, 106424 and 71424 of these volumes' groups.
@pytest.mark.parametrize("n,nz,dtype", [(30, 300000, "f32"), (28, 330000, "f32"), (56, 160000, "bf16")])
def test_volumes_of_many_rows(n, nz, dtype):
    """The rate and the threshold are exact; the maximum and most mismatches lie in the last rows."""
    import torch

    import __graft_entry__
    __graft_entry__.build()
    from paper_2211_03516_gb300 import inputs as I
    from paper_2211_03516_gb300 import vamrt as V
    w = I.TINY.scaled(nx=n, ny=n, nz=nz, voxel_mm=12.2 / n, nu=8, nv=8, n_angles=1)
    P = V.Projector.from_workload(w, I.workload_pupil(w))
    gen = torch.Generator(device="cuda:0").manual_seed(41)
    target = (torch.rand(w.vol_shape, device="cuda:0", generator=gen) < 0.5).float()
    dose = (0.2 + 0.5 * target).mul_(torch.rand(w.vol_shape, device="cuda:0", generator=gen).mul_(0.1).add_(0.95))
    tail = slice(nz - nz // 50, nz)
    dose[tail] = 1.7 - dose[tail]
    dose = dose.to({"f32": torch.float32, "bf16": torch.bfloat16}[dtype])
    ver, index = P.voxel_error_rate(dose, target)
    c = (np.arange(n) - 0.5 * (n - 1)) * w.voxel_mm
    resin = torch.from_numpy((c * c)[None, :] + (c * c)[:, None] <= w.r_inner_mm * w.r_inner_mm).to("cuda:0")
    # the rate is defined by FP32 bins of the stored dose
    x, f = dose.float()[:, resin].reshape(-1), target[:, resin].reshape(-1) > 0.5
    b = torch.floor(x * (1024.0 / x.max())).clamp_(0, 1023).long()
    below = torch.bincount(b[f], minlength=1024).cumsum(0)[:-1]
    above = (~f).sum() - torch.bincount(b[~f], minlength=1024).cumsum(0)[:-1]
    best = int((below + above).argmin())
    assert index == best + 1
    assert ver == float(below[best] + above[best]) / x.numel()
