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


@pytest.mark.parametrize("S,settings", [(40, {}), (40, dict(factor_ctas=152)), (40, dict(factor_ctas=8)),
                                        (250, dict(factor_ctas=152)), (250, dict(factor_ctas=9)), (250, dict(factor_ctas=6))])
def test_waits_that_give_up_leave_indices_in_bounds(S, settings):
    """Every wait gives up at once, over a workspace whose pivot lists have never been written: what is
    read there is kept in bounds, the launch ends at its barriers, the call reports the timeout; another
    column then solves as usual."""
    import numpy as np
    from paper_2512_06729_gb300 import synth, xk
    p = synth.small_column(S=S, L=9, n_two=4 * S, n_three=S, n_photo=5, W=40, elements="chons" if S < 110 else "full")
    col = xk.Column(p, "fp64", allocate=False, wait_polls=1, **settings)
    col.ws = torch.full((col.workspace_bytes + 256,), 0x7f, dtype=torch.uint8, device="cuda")
    col._call("xk_set_workspace", ctypes.c_void_p((col.ws.data_ptr() + 255) & ~255), ctypes.c_size_t(col.workspace_bytes))
    col.set_mixing_ratios(p.f0)
    n = col.get_state(device=True)
    for _ in range(2):
        with pytest.raises(xk.XkError) as err:
            col.step_delta(n, 1e-4)
        assert err.value.code == -7                # XK_ETIMEOUT
    torch.cuda.synchronize()
    a, b = xk.Column(p, "fp64", **settings), xk.Column(p, "fp64", twisted=0, factor_ctas=76)
    da, db = a.step_delta(n, 1e-4)[0], b.step_delta(n, 1e-4)[0]
    assert float(torch.linalg.norm(da - db) / torch.linalg.norm(db)) <= 1e-6
    for c in (col, a, b):
        c.close()


def test_a_column_that_timed_out_in_a_batch_runs_after_it():
    """A held barrier in a round: the slot's status says so, and out of the batch the column takes its
    step as if nothing had happened."""
    import numpy as np
    from paper_2512_06729_gb300 import synth, xk
    p = synth.small_column()
    b = xk.Batch(8 << 30, 2)
    col, other = (xk.Column(p, "fp64", factor_ctas=152, wait_polls=1 << 14) for _ in range(2))
    for c in (col, other):
        c.set_mixing_ratios(p.f0)
    n = other.get_state(device=True)
    slot = b.add(col, 1e-8)
    col.hold_next_barrier()
    b.step(1)
    assert b.poll(slot)[1:] == (True, -7)
    assert b.remove(slot) is col
    want = other.step_delta(n, 1e-4)[0].cpu().numpy()
    np.testing.assert_array_equal(col.step_delta(n, 1e-4)[0].cpu().numpy(), want)
    b.close()
