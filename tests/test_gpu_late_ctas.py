"""Steps whose grid does not fit on the device at once: a kernel of another stream holds most of the
SMs for some milliseconds, so that the other CTA pairs do the step and the remaining ones start
after the canvas has been scored.  They find the pass that the others worked on (the mask as it
was when the step began), nothing to do, and leave; the step's results are those of an undisturbed
one, and so are the next step's."""
import ctypes
import importlib.util
import os
import subprocess
import time

import pytest
import torch

import workloads as WL

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, never run there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from gpu_util import DeviceRunner  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HOLDER = r"""
#include <cuda_runtime.h>
// One block per SM (200 KB of shared memory each), each for `ns` nanoseconds.
__global__ void k_hold(unsigned long long ns) {
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    do {
        __nanosleep(1000);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    } while (t - t0 < ns);
}
extern "C" int hold_sms(int blocks, unsigned long long ns, void *stream) {
    cudaError_t e = cudaFuncSetAttribute(k_hold, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e == cudaSuccess) {
        k_hold<<<blocks, 32, 200 * 1024, static_cast<cudaStream_t>(stream)>>>(ns);
        e = cudaGetLastError();
    }
    return e;
}
"""
HOLD_NS = 60_000_000


@pytest.fixture(scope="module")
def hold_sms(tmp_path_factory):
    path = os.path.join(ROOT, "paper_2609_36452_gb300", "_build.py")
    spec = importlib.util.spec_from_file_location("_rpd_build_flags", path)
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    d = tmp_path_factory.mktemp("hold")
    (d / "hold.cu").write_text(HOLDER)
    lib = str(d / "libhold.so")
    subprocess.run([build.nvcc(), "-shared", "-Xcompiler", "-fPIC", str(d / "hold.cu"), "-o", lib] + build.ARCH,
                   check=True, capture_output=True)
    fn = ctypes.CDLL(lib).hold_sms
    fn.argtypes = [ctypes.c_int, ctypes.c_ulonglong, ctypes.c_void_p]
    return fn


class Held:
    """Steps of one context on a stream of their own, with `blocks` SMs held or none."""

    def __init__(self, hold_sms, runner, hidden, mask, blocks):
        self.hold_sms, self.runner, self.hidden, self.blocks = hold_sms, runner, hidden, blocks
        self.mask = mask.cuda().reshape(1, -1)
        self.side, self.main = torch.cuda.Stream(), torch.cuda.Stream()
        runner.ctx.set_stream(self.main)

    def timed(self, call, held):
        torch.cuda.synchronize()
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        if held:
            assert self.hold_sms(self.blocks, HOLD_NS, self.side.cuda_stream) == 0
            time.sleep(0.002)  # resident
        with torch.cuda.stream(self.main):
            t0.record()
            call()
            t1.record()
        torch.cuda.synchronize()
        return t0.elapsed_time(t1)

    def step(self, held):
        N = self.mask.shape[1]
        out = self.runner._alloc(1, N)
        ms = self.timed(lambda: self.runner.ctx.step(self.hidden, self.mask[0], 0.9, 1.0, out["commit"][0],
                                                     out["token"][0], out["stats"][0]), held)
        return ms, self.runner._fetch(out, self.mask, 1)[0]


def assert_equal(a, b):
    assert a["stats"] == b["stats"] and a["stats"]["status"] == 0
    for k in a:
        if k != "stats":
            assert (a[k] == b[k]).all(), k


# Of 152 SMs: 40 late pairs, and all but a few.
@pytest.mark.parametrize("blocks", [80, 136])
@pytest.mark.parametrize("N,masked,rule,projection", [
    (128, 3, "llada_block", "all"),   # the step finishes the first block: the mask then names the next one
    (1024, 961, "llada", "all"),      # 3844 rows; with any fewer another plan, of far more units
    (1024, 961, "llada", "lazy"),
    (300, 77, "llada", "auto"),
])
def test_late_pairs_find_the_pass_of_the_others(hold_sms, blocks, N, masked, rule, projection):
    K, d, V = 4, 256, 126464
    W, g = WL.make_head(V, d, 5, w_std=0.08)
    hidden = WL.make_hidden(W, K, N, 6, WL.u_profile(N, 0.5, 3.0), WL.calibrated_sigma(V, d, 0.08, 3.0),
                            flip_frac=0.1).hidden.cuda()
    mask = torch.zeros(N, dtype=torch.uint8)
    if rule == "llada_block":
        mask[:masked - 2] = 1  # at the confident end
        mask[32:] = 1
    else:
        mask[torch.randperm(N, generator=torch.Generator().manual_seed(7))[:masked]] = 1
    runner = DeviceRunner(W, g, K, rule=rule)
    try:
        runner.ctx.set_projection(projection)
        quiet = Held(hold_sms, runner, hidden, mask, 0)
        want = [quiet.step(False)[1] for _ in range(3)]
        if rule == "llada_block":
            assert want[0]["new_mask"][:32].sum() == 0 and want[0]["new_mask"].sum() == N - 32
        disturbed = Held(hold_sms, runner, hidden, mask, blocks)
        for i, held in enumerate([True, True, False]):
            ms, got = disturbed.step(held)
            assert_equal(want[i], got)
            assert ms < HOLD_NS * 1e-6 + 100, ms  # no wait ran out (2 s each)
    finally:
        runner.close()


def test_late_pairs_project_nothing_again(hold_sms):
    """A step takes no longer than the same pass without scoring, whose mask stays as it is."""
    K, d, V, N = 4, 1024, 126464, 1024
    gen = torch.Generator(device="cuda").manual_seed(9)
    W = (torch.randn(V, d, generator=gen, device="cuda") * 0.04).to(torch.bfloat16)
    hidden = torch.randn(K, N, d, generator=gen, device="cuda").to(torch.bfloat16)
    mask = torch.ones(N, dtype=torch.uint8)
    mask[:63] = 0  # 961 masked: 3844 rows in 304 units; 3840 rows would be 3705
    runner = DeviceRunner(W, torch.ones(d, dtype=torch.bfloat16), K)
    part = DeviceRunner(W, torch.ones(d, dtype=torch.bfloat16), K)
    try:
        part.ctx.set_vocab_shard(0, V)
        partials = torch.zeros(K, N, 4, device="cuda")
        passes = Held(hold_sms, part, hidden, mask, 136)
        call = lambda: part.ctx.step_shard_partials(hidden, passes.mask[0], partials)  # noqa: E731
        passes.timed(call, False)
        t_pass = min(passes.timed(call, True) for _ in range(3))
        Held(hold_sms, runner, hidden, mask, 0).step(False)
        t_step = min(Held(hold_sms, runner, hidden, mask, 136).step(True)[0] for _ in range(3))
    finally:
        runner.close()
        part.close()
    assert t_step < 1.4 * t_pass + 1, (t_step, t_pass)
