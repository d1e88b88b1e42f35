"""Optional scratch of low-degree FP32 meshes against a limit on device memory.

Uniform FP32 meshes of p <= 2 with many elements run two kernels through a scratch although they
could run one kernel without.  So no call that fits without that scratch may fail because of it.  The
library is linked again with cudaMalloc and cudaFree behind a counter with a limit (an allocation
beyond it returns cudaErrorMemoryAllocation; the device itself is never short of memory), and used in a
child process.

Bars: FP32 against FP64 of the same library 2e-6 (inputs rounded to float, short sums); end states of
a mixed solve to 1e-10 against the same solve without a limit 1e-8.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

COUNTER = r"""
#include <cstddef>
#include <map>
#include <mutex>
extern "C" int __real_cudaMalloc(void**, size_t);
extern "C" int __real_cudaFree(void*);
static std::mutex mu;
static std::map<void*, size_t> held;
static long long total = 0, limit = -1, refused = 0, peak = 0;
extern "C" int __wrap_cudaMalloc(void** p, size_t n) {
  std::lock_guard<std::mutex> g(mu);
  if (limit >= 0 && total + (long long)n > limit) {
    ++refused;
    return 2;  // cudaErrorMemoryAllocation
  }
  const int e = __real_cudaMalloc(p, n);
  if (e == 0) {
    held[*p] = n;
    total += (long long)n;
    if (total > peak) peak = total;
  }
  return e;
}
extern "C" int __wrap_cudaFree(void* p) {
  std::lock_guard<std::mutex> g(mu);
  auto it = held.find(p);
  if (it != held.end()) {
    total -= (long long)it->second;
    held.erase(it);
  }
  return __real_cudaFree(p);
}
extern "C" void mem_limit(long long n) { limit = n; }
extern "C" long long mem_total() { return total; }
extern "C" long long mem_peak() { return peak; }
extern "C" long long mem_refused() { return refused; }
"""

COMMON = r"""
import ctypes as C, sys
import numpy as np, torch
from paper_1307_5310_gb300 import meshgen, stm
stm.LIB_PATH = sys.argv[1]
L = stm.lib()
for f in ("mem_total", "mem_peak", "mem_refused"):
    getattr(L, f).restype = C.c_longlong
L.mem_limit.argtypes = [C.c_longlong]
dt = 0.01
m = meshgen.box_mesh(16, p=1, q=1)
meshgen.random_materials(m, 83, 84)
ne = 16 ** 3
test, tr, state = ne * 6 * 8, ne * 24 * 4, ne * 6 * 8
own = 4 * (test + tr)          # FP32 scratch of a direct apply
SRC = [dict(centre=(.5, .5, .5), dir=(0, 0, 1), sigma_x=.2, t0=.01, sigma_t=.05, amp=1.0)]

def slab(**kw):
    return stm.Slab(m, precision=stm.STM_MIXED, tol=1e-10, **kw)

def solve(s):
    s.set_state(u0)
    rc, rep = s.slab_solve(dt)
    assert rc == stm.STM_OK, rep
    return s.get_state()[0]

def apply32(s, ref):
    out.zero_()
    s.residual_apply(U.float(), out, 0.0, dt, prec=stm.STM_FP32)
    torch.cuda.synchronize()
    return float((out.double() - ref).norm() / ref.norm())

g = torch.Generator(device="cuda").manual_seed(5)
U = torch.empty(ne * 6 * 2 * 8, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=g)
u0 = torch.empty(state, dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=g)
out = torch.empty(test, dtype=torch.float32, device="cuda")
s = slab()
R = torch.empty(test, dtype=torch.float64, device="cuda")
s.residual_apply(U, R, 0.0, dt)
s.set_source_gauss(SRC)
RL = torch.empty_like(R)
s.residual_apply(U, RL, 0.0, dt)
s.close()
# a mixed solve without a direct FP32 apply: the bytes it takes beyond the context
s = slab()
base = L.mem_total()
ref = solve(s)
need = L.mem_total() - base
s.close()
"""

CASES = {
    # nothing but the solver's vectors, the FP64 scratch and the small GMRES state
    "solve_takes_no_fp32_scratch": r"""
ldv = (test + 63) // 64 * 64
assert need <= 8 * 2 * test + 4 * 11 * ldv + 4 * test + 8 * (test + tr) + 16384, need
""",
    # a direct FP32 apply first; the solve then fits only if that apply's scratch is given back
    "solve_after_apply": r"""
s = slab()
assert apply32(s, R) < 2e-6
assert L.mem_total() - base <= own + 4096
L.mem_limit(base + need + 65536)
u = solve(s)
assert np.linalg.norm(u - ref) < 1e-8 * np.linalg.norm(ref)
assert apply32(s, R) < 2e-6
n = L.mem_refused()
assert apply32(s, R) < 2e-6 and L.mem_refused() == n   # not tried again
""",
    "load_after_apply": r"""
s = slab()
assert apply32(s, R) < 2e-6
L.mem_limit(L.mem_total() - own + 12 * test + 65536)
s.set_source_gauss(SRC)
assert apply32(s, RL) < 2e-6
""",
    # the FP64 half of the load fits, the FP32 half does not: refused, and again, until there is room
    "load_in_halves": r"""
s = slab()
s.residual_apply(U, R, 0.0, dt)
s.set_source_gauss(SRC)
L.mem_limit(L.mem_total() + 8 * test + 4096)
n = L.mem_total()
for k in range(2):
    try:
        apply32(s, RL)
        assert False, "fits"
    except stm.StmError as e:
        assert e.code == stm.STM_ENOMEM, e
    assert L.mem_total() == n
L.mem_limit(-1)
assert apply32(s, RL) < 2e-6
""",
    # no room at all: the apply runs without scratch, asks for it once and leaves no error text
    "apply_without_room": r"""
s = slab()
L.mem_limit(L.mem_total())
assert apply32(s, R) < 2e-6
assert apply32(s, R) < 2e-6
assert L.mem_refused() == 1, L.mem_refused()
assert L.stm_last_error(s.ctx) == b""
""",
    # a captured apply holds no scratch of the context: it survives the scratch being given back
    "captured_apply": r"""
side = torch.cuda.Stream()
s = slab(stream=side.cuda_stream)
u32 = U.float()
torch.cuda.synchronize()
s.residual_apply(u32, out, 0.0, dt, prec=stm.STM_FP32)
torch.cuda.synchronize()
gr = torch.cuda.CUDAGraph()
with torch.cuda.graph(gr, stream=side):
    s.residual_apply(u32, out, 0.0, dt, prec=stm.STM_FP32)
gr.replay()
torch.cuda.synchronize()
one = out.clone()
L.mem_limit(base + need + 65536)
solve(s)
out.zero_()
torch.cuda.synchronize()
gr.replay()
torch.cuda.synchronize()
assert torch.equal(out, one)
assert float((out.double() - R).norm() / R.norm()) < 2e-6
""",
    # the server admits such a request by what its solve takes
    "server_footprint": r"""
srv = stm.Server(workers=1, precision=stm.STM_MIXED, tol=1e-8)
r, _ = srv.wait(srv.submit(16, 1, 1, 1, dt))
assert r["status"] == stm.STM_OK
ldv = (test + 63) // 64 * 64
assert r["footprint_bytes"] <= 8 * (test + tr) + 16 * state + 24 * test + 4 * test * 13 + ne * 512 + (64 << 20)
assert L.mem_peak() - L.mem_total() <= r["footprint_bytes"]
srv.close()
""",
}


@pytest.fixture(scope="module")
def lib_path(tmp_path_factory):
    import __graft_entry__

    __graft_entry__.build()
    from paper_1307_5310_gb300 import build

    d = tmp_path_factory.mktemp("counted")
    src, so = d / "counter.cpp", d / "libstm_counted.so"
    src.write_text(COUNTER)
    objs = [os.path.join(build.BUILD, obj) for _, obj, _ in build._units()]
    subprocess.run(["g++", "-O1", "-fPIC", "-c", str(src), "-o", str(d / "counter.o")], check=True)
    subprocess.run([build._nvcc(), *build.ARCH, "-shared", "-Xlinker", "--wrap=cudaMalloc", "-Xlinker",
                    "--wrap=cudaFree", "-o", str(so), *objs, str(d / "counter.o")], check=True)
    return str(so)


@pytest.mark.parametrize("case", sorted(CASES))
def test_low_degree_fp32_memory(lib_path, case):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", COMMON + CASES[case], lib_path], cwd=root, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
