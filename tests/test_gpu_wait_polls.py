"""cfg.wait_polls governs the waits between the CTAs of a cluster as it does those between the CTAs of a
grid: a wait for something that never arrives gives up after that many polls, and says so."""
import ctypes
import os
import subprocess
import time

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "xk_mbar.cuh"
__global__ void __cluster_dims__(2, 1, 1) k(xk::Ctl *ctl)
{
    __shared__ unsigned long long bar;
    if (threadIdx.x == 0) {
        xk::mbar_init(xk::smem_u32(&bar));
        xk::mbar_wait(xk::smem_u32(&bar), 0u, ctl);      // nothing arrives
    }
}
extern "C" int run(unsigned long long polls)
{
    xk::Ctl h = {}, *d = nullptr;
    h.wait_polls = polls;
    if (cudaMalloc(&d, sizeof h) != cudaSuccess) return -1;
    cudaMemcpy(d, &h, sizeof h, cudaMemcpyHostToDevice);
    k<<<2, 1>>>(d);
    const cudaError_t e = cudaMemcpy(&h, d, sizeof h, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? h.err_timeout : -1;
}
"""


def test_a_cluster_wait_gives_up_after_the_configured_polls(tmp_path):
    """Ten thousand polls of a barrier that stays open end within a fifth of a second; the default's are
    four hundred times as many."""
    from paper_2512_06729_gb300 import build as xkbuild
    src, out = tmp_path / "wait.cu", tmp_path / "libwait.so"
    src.write_text(SOURCE)
    subprocess.run([xkbuild.nvcc(), *xkbuild.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-I", xkbuild.CSRC, "-I", os.path.join(xkbuild.HERE, "..", "include"),
                    str(src), "-o", str(out)], check=True)
    run = ctypes.CDLL(str(out)).run
    run.argtypes = [ctypes.c_ulonglong]
    assert run(8) == 1
    t0 = time.perf_counter()
    assert run(10000) == 1
    t = time.perf_counter() - t0
    assert t < 0.2


@pytest.mark.parametrize("ctas", [152, 8])
def test_two_chains_of_the_elimination_time_out_and_recover(ctas):
    """The grid barriers of both chains held: their flags and clusters' waits run on, every CTA leaves at
    the layer's end, the call reports the timeout and the next solves normally."""
    import numpy as np
    from oracle.oracle import Oracle
    from paper_2512_06729_gb300 import synth, xk
    p = synth.small_column()
    o = Oracle(p)
    n = o.initial_state()
    s = np.maximum(n, 1e-20 * o.grid()[0][:, None])
    ref = o.step_delta(n, 1e-4)
    nd = torch.as_tensor(n, device="cuda")
    col = xk.Column(p, "fp64", factor_ctas=ctas, twisted=1, wait_polls=1 << 14)
    for held in (False, True, False, True, False):
        if held:
            col.hold_next_barrier()
            with pytest.raises(xk.XkError) as err:
                col.step_delta(nd, 1e-4)
            assert err.value.code == -7            # XK_ETIMEOUT
        else:
            d, _, _ = col.step_delta(nd, 1e-4)
            assert np.max(np.abs(d.cpu().numpy() - ref) / s) < 1e-8
    col.close()
