"""The first calls of a process made by several threads at once: each takes the path it would take alone.  (What a process looks up
once, the driver's tensor map encoder among it, must not be taken for missing while another thread is still looking it up.)"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

# threads that leave a spin barrier together, which threads of the interpreter do not
TOGETHER = r"""
#include <atomic>
#include <cstddef>
#include <thread>
#include <vector>
typedef int (*forward)(void *, void *, void *, void *, void *, void *, void *, void *, void *, void *, size_t, void *);
typedef int (*read_status)(void *, void *, void *, unsigned *);
extern "C" void together(forward fn, read_status warm, int n, void **a, size_t ws_bytes, int *rc) {
    std::atomic<int> here{0};
    std::vector<std::thread> threads;
    for (int i = 0; i < n; ++i)
        threads.emplace_back([&, i] {
            void **x = a + 11 * i;
            unsigned bits = 0;
            warm(x[0], x[9], x[10], &bits);               // the thread's first CUDA calls
            here.fetch_add(1);
            while (here.load() < n) {}
            rc[i] = fn(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7], x[8], x[9], ws_bytes, x[10]);
        });
    for (auto &t : threads) t.join();
}
"""

SCRIPT = r"""
import ctypes, sys
import torch
from paper_2106_09236_b200 import binding as ps
N, B, H, T = 6, 1, 2, 300
lib, helper = ps.load(), ctypes.CDLL(sys.argv[1])
q = torch.randn((B, H, T, 64), device="cuda").bfloat16()
lengths = torch.full((B,), T, dtype=torch.int32, device="cuda")
keep, args = [], []
for n in range(N):
    plan = ps.Plan(B, H, T, path=ps.PSATTN_PATH_FUSED)
    idx = torch.zeros((B, T, plan.idx_cols), dtype=torch.int32, device="cuda")
    O, sel, st = torch.empty_like(q), torch.empty((B, H, plan.u_max), dtype=torch.int32, device="cuda"), torch.cuda.Stream()
    keep.append((plan, idx, O, sel, st))
    args += [plan.handle.value] + [x.data_ptr() for x in (q, q, q, lengths, idx, O, sel)] + [None, plan.workspace.data_ptr(), st.cuda_stream]
torch.cuda.synchronize()
rc = (ctypes.c_int * N)(*[-1] * N)
address = lambda f: ctypes.cast(f, ctypes.c_void_p)
helper.together(address(lib.psattn_forward), address(lib.psattn_read_status), N, (ctypes.c_void_p * len(args))(*args),
                ctypes.c_size_t(keep[0][0].workspace_bytes), rc)
torch.cuda.synchronize()
assert list(rc) == [0] * N, list(rc)
"""


def test_first_forward_calls_of_six_threads(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    (tmp_path / "together.cpp").write_text(TOGETHER)
    helper = str(tmp_path / "together.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", str(tmp_path / "together.cpp"), "-o", helper])
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", SCRIPT, helper], cwd=root, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
