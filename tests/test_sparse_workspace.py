"""The sparse solver's workspace after a failed allocation, on the CPU.

Its allocation code is compiled against fakes of the CUDA calls, one of which
fails: the call must report it, and the next call must find or make every
buffer instead of going on without the one that was missing."""

import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include "la.h"
typedef int cudaError_t;
typedef int cudaEvent_t;
enum { cudaSuccess = 0, cudaDevAttrMultiProcessorCount = 16 };
static int calls, failing;
static int fake() { return ++calls == failing ? 2 : 0; }
template <class T> int cudaMalloc(T **p, size_t n) { if (fake()) return 2; *p = (T *)malloc(n); return 0; }
template <class T> int cudaMallocHost(T **p, size_t n) { return cudaMalloc(p, n); }
static int cudaFree(void *p) { free(p); return 0; }
static int cudaGetDevice(int *d) { *d = 0; return fake(); }
static int cudaDeviceGetAttribute(int *v, int, int) { if (fake()) return 2; *v = 152; return 0; }
static int cudaEventCreate(cudaEvent_t *e) { if (fake()) return 2; *e = 7; return 0; }
template <class F> int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *o, F, int, int) { *o = 4; return 0; }
template <bool Z> void k_sp_refine() {}
constexpr int kBlock = 256;
struct Ctrl { int x; };
struct FinCtrl { int x; };
@CODE@
int main() {
    int reported = 0;
    for (failing = 1; failing <= 40; ++failing) {
        const int k = failing;
        SparseWorkspace w;
        w.ev[0] = w.ev[1] = 0;
        calls = 0;
        const la_status first = ensure_sws(w, 5000);
        const bool hit = calls >= k;
        if (hit != (first != LA_OK)) return printf("failure %d was not reported\n", k), 1;
        reported += hit;
        failing = 0;
        if (ensure_sws(w, 5000) != LA_OK) return printf("no recovery after failure %d\n", k), 1;
        failing = k;
        if (!w.key || !w.qm || !w.colseen || !w.pot || !w.rowcol || !w.rows || !w.fin || !w.ctrl || !w.h_ctrl ||
            w.num_sms != 152 || w.occ != 4 || w.ev[0] != 7 || w.ev[1] != 7 || w.cap < 5000)
            return printf("something is missing after failure %d\n", k), 1;
    }
    return reported >= 10 ? 0 : (printf("only %d failures\n", reported), 1);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="g++ not found")
def test_every_failed_allocation_is_made_good_by_the_next_call(tmp_path):
    src = open(os.path.join(ROOT, "paper_1110_6231_gb300", "csrc", "la_sparse.cu")).read()
    struct = re.search(r"^struct SparseWorkspace \{.*?^\};\n", src, re.S | re.M).group(0)
    ensure = re.search(r"^la_status ensure_sws\(.*?^\}\n", src, re.S | re.M).group(0)
    cpp = tmp_path / "ws.cpp"
    cpp.write_text(HARNESS.replace("@CODE@", struct + ensure))
    exe = str(tmp_path / "ws")
    subprocess.run(["g++", "-std=c++17", "-I" + os.path.join(ROOT, "include"), str(cpp), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
