"""Plans on a device with little memory left: the tables and the scratch that only make the FP64
contractions and the lattice transforms faster may fail to allocate, and the kernels that need
none of them take their place.  The planning code of both runs here on the host against
counting stand-ins for the three memory calls, the n-th allocation failing.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1911_05633_gb300", "csrc")

SOURCE = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <cstdlib>
#include <set>
static int g_calls = 0, g_fail = 0;
static std::set<void*> g_live;
static cudaError_t test_malloc(void** p, size_t) {
  if (++g_calls == g_fail) return cudaErrorMemoryAllocation;
  *p = std::malloc(1);
  g_live.insert(*p);
  return cudaSuccess;
}
static cudaError_t test_free(void* p) {
  if (p && !g_live.erase(p)) std::printf("freed twice\n");
  std::free(p);
  return cudaSuccess;
}
static cudaError_t test_memcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
template <typename F> static cudaError_t test_raise(F*, size_t) { return cudaSuccess; }
#include "smem_limit.h"
#define cudaMalloc test_malloc
#define cudaFree test_free
#define cudaMemcpy test_memcpy
#define raise_smem_limit test_raise
#include "kernels_lattice.cu"
#include "kernels_chain.cu"
namespace gw {
void set_last_error(const std::string&) {}
KernelTimer*& current_timer() { static KernelTimer* t = nullptr; return t; }
}
int main() {
  gw::HostPlan h;
  h.n_species = 1;
  h.n_orb = {9};
  h.n_prod = {16};
  h.C.assign(1, std::vector<double>(16 * 81, 0.5));
  h.n_atoms = 1;
  h.species = {0};
  h.orb_off = {0, 9};
  h.pb_off = {0, 16};
  h.n_k = 3;
  h.n_tau = 5;
  h.entries.assign(8 * 3, 0);
  h.pair_start = {0, 3};
  h.phase.assign(2 * 9, 0.5);
  for (int fail = 0; fail < 20; ++fail) {
    g_fail = fail;
    g_calls = 0;
    gw::ChainPlan c;
    gw::chain_init(c, h);
    const int tables = g_calls;
    const bool s = c.ok && gw::chain_alloc_s(c, h, 1 << 20) == GW_OK, p = c.ok && gw::chain_alloc_p(c, h, 1 << 20) == GW_OK;
    const int all = g_calls;
    std::printf("chain %d %d %d: %d %d %d %d\n", fail, tables, all, c.ok, s == c.s_ready ? s : -1, p == c.p_ready ? p : -1,
                c.s_ready || (!c.d_AS && !c.d_eS && !c.d_D));
    gw::chain_free(c);
    g_calls = 0;
    gw::LatticePlan l;
    gw::lattice_init(l, h);
    std::printf("lattice %d %d: %d\n", fail, g_calls, l.ok);
    gw::lattice_free(l);
    if (!g_live.empty()) std::printf("left behind %zu\n", g_live.size());
  }
  return 0;
}
"""


def test_failed_allocations_leave_the_plan_usable(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "alloc.cu", tmp_path / "alloc"
    src.write_text(SOURCE)
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "-I", CSRC, "-I",
                        os.path.join(CSRC, "..", "..", "include"), str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True).stdout.splitlines()
    assert len(out) == 40, out
    full = [line.split() for line in out[:2]]  # nothing fails
    assert full[0][4:] == ["1", "1", "1", "1"] and full[1][3] == "1"
    tables, every = int(full[0][2]), int(full[0][3][:-1])
    for line in out[2:]:
        w = line.split()
        fail = int(w[1])
        if w[0] == "lattice":
            assert w[3] == ("0" if fail <= int(full[1][2][:-1]) else "1"), line
        else:
            ok = fail > tables
            # the first of Sigma's three buffers comes after the tables, then P's two
            s = ok and not (tables < fail <= tables + 3)
            n = int(w[3][:-1])
            p = ok and not (s and tables + 3 < fail <= every)
            assert w[4:] == [str(int(ok)), str(int(s)), str(int(p)), "1"], (line, tables, every, n)
