"""A router kernel starts, and brings rows of its input into L2, while the kernel before it still runs - if that kernel allows
it.  Here that kernel allows it first thing, waits, and only then writes the rows: the call must see what it wrote.
"""
import ctypes
import subprocess

import pytest
import torch

from paper_2608_14205_b200 import binding as B
from paper_2608_14205_b200 import build
from paper_2608_14205_b200 import inputs as I
from tests import parity_util as P

pytestmark = pytest.mark.gpu

# On 40 SMs: a router block takes nearly all registers of one, so the call's blocks start on the others.
LATE_WRITER = r"""
#include <cuda_runtime.h>
__global__ void __launch_bounds__(256) late_copy(const uint4* a, uint4* to_a, const uint4* b, uint4* to_b, long long n, int cycles) {
  asm volatile("griddepcontrol.launch_dependents;");
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) {}
  for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += gridDim.x * 256ll) { to_a[i] = a[i]; to_b[i] = b[i]; }
}
extern "C" int write_late(const void* a, void* to_a, const void* b, void* to_b, long long n16, int cycles, void* stream) {
  if (cycles < 0 || cycles > 1000000) return 1;
  late_copy<<<40, 256, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<const uint4*>(a), static_cast<uint4*>(to_a),
                                                                static_cast<const uint4*>(b), static_cast<uint4*>(to_b), n16, cycles);
  return cudaGetLastError() == cudaSuccess ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def write_late(tmp_path_factory):
    at = tmp_path_factory.mktemp("late_writer")
    (at / "late.cu").write_text(LATE_WRITER)
    subprocess.run([build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O2", "-shared", "-Xcompiler", "-fPIC",
                    "-o", str(at / "late.so"), str(at / "late.cu")], check=True, capture_output=True)
    fn = ctypes.CDLL(str(at / "late.so")).write_late
    fn.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_longlong, ctypes.c_int, ctypes.c_void_p]
    return fn


@pytest.mark.parametrize("name,T,pair_limit", [("tiny", 300, 0), ("qwen3", 2000, 0), ("qwen3", 8192, 0), ("dsv3", 1500, 0),
                                               ("dsv3", 1500, 2)])
@pytest.mark.parametrize("call", ["plan", "layer"])
def test_rows_written_after_the_call_may_start_are_the_ones_it_uses(write_late, name, T, pair_limit, call):
    wl = I.WORKLOADS[name]
    layers = [I.make_layer(wl, l, 0, T=T) for l in range(2)]
    ctx = P.make_context(wl, T)
    ctx.fb_set_pair_limit(pair_limit)
    dev = torch.device("cuda", ctx.device)
    sb = layers[0].select_bias.to(dev) if layers[0].select_bias is not None else None
    router = B.make_router(layers[0].W.to(dev), None, sb)
    pi = layers[0].expert_to_slot.to(dev)
    budget = B.make_budget(**P.budget_kwargs(wl, T))
    src = [(li.h_prev.to(dev), li.H.to(dev)) for li in layers]
    x, H = torch.zeros_like(src[0][0]), torch.zeros_like(src[0][1])
    i32 = lambda n: torch.full((max(1, n),), -3, dtype=torch.int32, device=dev)

    def run(a, b):
        o = [i32(wl.E), i32(wl.E), i32(4 * (wl.E // 2)).zero_(), i32(1), i32(wl.R), i32(wl.R)]
        if call == "plan":
            return lambda: ctx.fb_predict_and_plan(router, a, T, pi, budget, 0, *o), o
        o += [i32(T * wl.k), torch.zeros(T * wl.k, device=dev), i32(wl.E + 1), i32(wl.R + 1), i32(T * wl.k), i32(T * wl.k), i32(wl.R)]
        return lambda: ctx.fb_layer_step(router, a, b, T, pi, budget, 0, *o), o

    want = []
    for a, b in src:
        go, o = run(a, b)
        go()
        want.append(o)
    calls = [run(x, H) for _ in range(8)]
    torch.cuda.synchronize(dev)
    stream = torch.cuda.current_stream(dev).cuda_stream
    for i, (go, _) in enumerate(calls):
        a, b = src[i % 2]
        # up to 100 us between "the next may start" and the first write: long enough for all that a call may bring in
        assert write_late(a.data_ptr(), x.data_ptr(), b.data_ptr(), H.data_ptr(), x.numel() // 8, (20000, 200000)[i // 2 % 2], stream) == 0
        go()
    torch.cuda.synchronize(dev)
    assert ctx.fb_device_status() == 0
    for i, (_, o) in enumerate(calls):
        for j, (got, ref) in enumerate(zip(o, want[i % 2])):
            assert torch.equal(got, ref), (i, j)
    ctx.close()
