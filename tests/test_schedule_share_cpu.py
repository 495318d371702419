"""Plans that share the columns' last planes among the CTAs left over (plan_persistent with
`share`), on the CPU: every plane of every tile column is computed once, over plane counts and
column counts around those where the candidate starts and ends to apply."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")
CHECK = r"""
#include <cstdio>
#include <vector>
#include "step3d.h"
int main()
{
    int other = 0;
    for (int M : {4, 8})
        for (int nz = 1; nz <= 330; nz += nz < 80 ? 1 : 11)
            for (int columns : {1, 2, 33, 56, 75, 76, 77, 90, 95, 101, 102, 138, 151, 152, 153, 303, 304, 305}) {
                fwi::Step3dParams p{}, q{};
                p.M = q.M = M;
                p.nz = q.nz = nz;
                const int grid = fwi::plan_persistent(p, columns, 304, true, true);
                fwi::plan_persistent(q, columns, 304, true, false);
                if (p.zfirst != q.zfirst) ++other;
                std::vector<int> seen((size_t)columns * nz, 0);
                for (int k = 0; k < grid; ++k) {
                    int col, z0, z1;
                    for (int i = 0; fwi::schedule_segment(p, columns, k, i, &col, &z0, &z1); ++i) {
                        if (col < 0 || col >= columns || z0 < 0 || z1 > nz || z0 >= z1) return 1;
                        for (int z = z0; z < z1; ++z) ++seen[(size_t)col * nz + z];
                    }
                }
                if (grid < 1 || grid > 304) return 2;
                for (int s : seen)
                    if (s != 1) return 3;
            }
    std::printf("ok %d\n", other);
    return 0;
}
"""


def test_shared_last_planes_cover_every_plane_once(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("g++ and the CUDA headers are needed to build the check")
    csrc = os.path.join(ROOT, "paper_1912_08063_gb300", "csrc")
    src, exe = tmp_path / "share.cpp", str(tmp_path / "share")
    src.write_text(CHECK)
    r = subprocess.run([cxx, "-O2", "-std=c++17", f"-I{CUDA}/include", f"-I{ROOT}/include", f"-I{csrc}", str(src),
                        os.path.join(csrc, "tmap.cpp"), f"-L{CUDA}/lib64", "-lcudart", "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    env = dict(os.environ, LD_LIBRARY_PATH=f"{CUDA}/lib64:" + os.environ.get("LD_LIBRARY_PATH", ""))
    out = subprocess.run([exe], capture_output=True, text=True, env=env, timeout=120)
    assert out.returncode == 0 and int(out.stdout.split()[1]) > 50, (out.returncode, out.stdout)
