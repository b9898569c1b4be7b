"""The host's schedule of a digit-product item (dg_schedule in csrc/gke_digits.cuh),
compiled for the CPU: what exceeds the kernel's tables or the four terms up to which
its FP32 sums are exact is refused; otherwise every term's B field is in its slot
when it runs, each slot is released before it is loaded again, and all are released
at the end of an item."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_06409_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

SOURCE = r"""
#include <cstdio>
#include "gke_digits.cuh"
using namespace gke;
static std::vector<std::vector<HostTerm>> jobs(int n, int nt, int nb)
{
    std::vector<std::vector<HostTerm>> v(n);
    for (int j = 0, f = 0; j < n; ++j)
        for (int t = 0; t < nt; ++t, ++f) v[j].push_back({f % 20, (f * 7 + j) % nb, (f & 1) != 0});
    return v;
}
static bool sound(const DgArgs& a, const std::vector<std::vector<HostTerm>>& js)
{
    int held[DG_NB], q = 0;
    bool busy[DG_NB];
    for (int i = 0; i < DG_NB; ++i) { held[i] = -1; busy[i] = false; }
    for (size_t j = 0; j < js.size(); ++j) {
        if (a.job[j].nt != js[j].size() || a.job[j].step != q) return false;
        for (int pass = 0; pass < 2; ++pass)
            for (size_t t = 0; t < js[j].size(); ++t, ++q) {
                const DgStep& s = a.step[q];
                if (s.fa != js[j][t].fa || s.fb != js[j][t].fb || ((s.flags & DF_NEG) != 0) != js[j][t].neg) return false;
                if (((s.flags & DF_FIRST) != 0) != (t == 0) || ((s.flags & DF_LAST) != 0) != (t + 1 == js[j].size()) ||
                    ((s.flags & DF_HI) != 0) != (pass == 1)) return false;
                if (s.flags & DF_LOAD) {
                    if (busy[s.slot]) return false;
                    busy[s.slot] = true;
                    held[s.slot] = s.fb;
                }
                if (!busy[s.slot] || held[s.slot] != s.fb) return false;
                if (s.flags & DF_FREE) busy[s.slot] = false;
            }
    }
    for (int i = 0; i < DG_NB; ++i) if (busy[i]) return false;
    return q == a.nstep;
}
int main()
{
    static DgArgs a;
    const int shapes[][3] = {{1, 1, 1}, {8, 3, 5}, {13, 4, 20}, {20, 2, 20}, {14, 4, 3}, {18, 3, 9}};
    for (auto& s : shapes) {
        auto js = jobs(s[0], s[1], s[2]);
        if (!dg_schedule(a, js) || !sound(a, js)) { printf("unsound %d %d %d\n", s[0], s[1], s[2]); return 1; }
    }
    if (dg_schedule(a, jobs(1, 5, 3))) { printf("five terms\n"); return 1; }
    if (dg_schedule(a, jobs(1, 0, 3))) { printf("no term\n"); return 1; }
    if (dg_schedule(a, jobs(21, 1, 3))) { printf("contractions\n"); return 1; }
    if (dg_schedule(a, jobs(15, 4, 3))) { printf("steps\n"); return 1; }
    printf("ok\n");
    return 0;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="nvcc not installed")
def test_schedule(tmp_path):
    src, exe = tmp_path / "schedule.cu", tmp_path / "schedule"
    src.write_text(SOURCE)
    subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", CSRC, "-o", str(exe), str(src)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
