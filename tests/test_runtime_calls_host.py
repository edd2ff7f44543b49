"""What the library asks of the CUDA runtime, on a fake runtime of two devices (fake_cuda_runtime.cpp):
the built objects are linked against it, device memory is host memory and kernels do nothing."""
import ctypes
import os
import subprocess
import types

import numpy as np
import pytest

from paper_2512_06729_gb300 import build as xkbuild
from paper_2512_06729_gb300 import synth, xk

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    pytest.importorskip("torch")
    xkbuild.build()
    out = str(tmp_path_factory.mktemp("fake") / "libxk_fake.so")
    objs = [os.path.join(xkbuild.BUILD, s.replace(".cu", ".o")) for s in xkbuild.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        xkbuild.build(force=True)
    symbols = subprocess.run(["nm", "-u", *objs], capture_output=True, text=True, check=True).stdout
    linked = {w for w in symbols.split() if w.startswith("__cudaRegisterLinkedBinary")}
    include = os.path.join(os.path.dirname(os.path.dirname(xkbuild.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-Wl,-Bsymbolic", "-I", include, "-o", out,
                    os.path.join(HERE, "fake_cuda_runtime.cpp"), *objs,
                    *(f"-Wl,--defsym={s}=fake_linked_binary" for s in linked)], check=True)
    lib = ctypes.CDLL(out)
    for name, (res, args) in xk.SIGNATURES.items():
        f = getattr(lib, name)
        f.restype, f.argtypes = res, args
    lib.fake_refused.restype = ctypes.c_char_p
    return lib


@pytest.fixture
def column(fake, monkeypatch):
    """column(problem, precision, device, **settings): a context with its workspace in host memory."""
    monkeypatch.setattr(xk, "_lib", fake)
    made = []

    def make(p, precision, device, **kw):
        c = xk.Column(p, precision, device=device, stream=types.SimpleNamespace(cuda_stream=0), allocate=False, **kw)
        c.ws = np.zeros(c.workspace_bytes + 256, np.uint8)
        base = (c.ws.ctypes.data + 255) & ~255
        c._call("xk_set_workspace", ctypes.c_void_p(base), ctypes.c_size_t(c.workspace_bytes))
        made.append(c)
        return c

    yield make
    for c in made:
        c.close()


def _step(col):
    n, d = np.zeros((col.L, col.S)), np.zeros((col.L, col.S))
    it, resid = ctypes.c_int(), ctypes.c_double()
    col._call("xk_step_delta", ctypes.c_void_p(n.ctypes.data), 1e-4, ctypes.c_void_p(d.ctypes.data), ctypes.byref(it),
              ctypes.byref(resid))


_PROBLEMS = {
    "small": lambda: synth.small_column(L=12),
    "chons": lambda: synth.chons_column(L=20),
    "full": lambda: synth.full_column(L=6),
}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name", list(_PROBLEMS))
def test_every_device_of_a_process_runs_a_step(fake, column, name, precision):
    """Contexts on two devices of one process, in both orders of creation and use: every kernel's
    shared-memory limit is raised where it is launched, and persistent grids fit the device's own SMs."""
    p = _PROBLEMS[name]()
    first = column(p, precision, 0)
    _step(first)
    second = column(p, precision, 1)
    before = fake.fake_launches(1)
    _step(second)
    _step(first)
    _step(second)
    assert fake.fake_refused() == b""
    assert fake.fake_launches(1) > before


def _batch(fake, column, slots, columns, p, precision):
    b = xk.Batch(1 << 40, slots)
    for _ in range(columns):
        b.add(column(p, precision, 0), 1e-8)
    return b


@pytest.mark.parametrize("how,precision,slots,columns,nodes", [
    ("round", "mixed", 8, 8, True), ("round", "mixed", 16, 8, True), ("round", "mixed", 9, 9, False),
    ("submit", "mixed", 8, 2, True), ("submit", "mixed", 9, 2, False),
    ("round", "fp64", 8, 2, True), ("submit", "fp64", 6, 2, True), ("submit", "fp64", 7, 2, False)])
def test_columns_of_a_batch_do_not_wait_for_connections(fake, column, how, precision, slots, columns, nodes):
    """Steps captured with conditional nodes run on the device's connections, eight by default: no more
    columns than that are captured with them."""
    S = 40 if precision == "mixed" else 160          # the FP64 elimination: the reduction has no nodes
    p = synth.small_column(S=S, L=9, n_two=3 * S, n_three=S, elements="chons" if S < 110 else "full")
    b = _batch(fake, column, slots, columns, p, precision)
    before = fake.fake_conditional_nodes()
    if how == "round":
        b.step(1)
    else:
        b.submit(0, 1)
    assert (fake.fake_conditional_nodes() > before) == nodes
    b.close()


def _launches_of(fake, name):
    grid, cluster = ctypes.c_int(), ctypes.c_int()
    n = fake.fake_launches_of(name.encode(), ctypes.byref(grid), ctypes.byref(cluster))
    return n, grid.value, cluster.value


# (species, CTAs) -> kernel, its grid and cluster: shared-memory columns where they fit, else the cluster
# that leaves each of two chains the most CTAs
@pytest.mark.parametrize("S,ctas,kernel,grid,cluster", [
    (40, 2, "k_factor64I", 2, 1), (40, 4, "k_factor64_flow", 4, 1), (96, 8, "k_factor64_flow", 8, 2),
    (250, 2, "k_factor64I", 2, 1), (250, 4, "k_factor64I", 4, 2), (250, 6, "k_factor64I", 6, 1),
    (250, 9, "k_factor64_flow", 8, 1), (250, 19, "k_factor64_flow", 16, 4), (400, 8, "k_factor64I", 8, 4),
    (400, 16, "k_factor64_flow", 16, 2),
    (594, 3, "k_factor64I", 2, 1), (594, 4, "k_factor64I", 4, 2), (594, 6, "k_factor64I", 6, 1), (594, 9, "k_factor64I", 8, 4),
    (594, 12, "k_factor64I", 12, 2), (594, 38, "k_factor64_flow", 36, 2), (594, 152, "k_factor64_flow", 152, 4)])
def test_elimination_on_few_ctas_keeps_them_busy(fake, column, S, ctas, kernel, grid, cluster):
    p = synth.small_column(S=S, L=4, n_two=2 * S, n_three=S // 2, n_photo=5, W=40, elements="chons" if S < 110 else "full")
    col = column(p, "fp64", 0, factor_ctas=ctas)
    fake.fake_forget_launches()
    _step(col)
    assert _launches_of(fake, "k_factor64")[0] == 2
    assert _launches_of(fake, kernel) == (2, grid, cluster)


@pytest.mark.parametrize("S,slots,reduction", [(64, 64, True), (80, 64, False), (96, 16, True), (96, 32, True), (96, 64, False), (120, 4, True),
                                               (152, 4, True), (152, 5, False), (152, 64, False)])
def test_small_shares_take_the_elimination(fake, column, S, slots, reduction):
    """The FP64 route of a column in a batch goes by its share of the SMs; alone, before and after, it is
    the reduction at these sizes."""
    p = synth.small_column(S=S, L=9, n_two=2 * S, n_three=S // 2, n_photo=5, W=40, elements="chons" if S < 110 else "full")
    b = xk.Batch(1 << 40, slots)
    col = column(p, "fp64", 0)
    slot = b.add(col, 1e-8)
    fake.fake_forget_launches()
    b.step(1)
    assert (_launches_of(fake, "k_inv64")[0] > 0) == reduction
    assert (_launches_of(fake, "k_factor64")[0] > 0) == (not reduction)
    b.remove(slot)
    fake.fake_forget_launches()
    _step(col)
    assert _launches_of(fake, "k_inv64")[0] > 0 and _launches_of(fake, "k_factor64")[0] == 0
    b.close()


@pytest.mark.parametrize("how", ["round", "submit", "run"])
def test_no_conditional_nodes_under_mps(fake, column, how):
    """Cooperative kernels, which the conditional parts hold, may stand in conditional nodes only while
    the device is not shared through MPS: there the steps are captured without such nodes."""
    fake.fake_set_mps(1)
    b = _batch(fake, column, 2, 1, synth.small_column(L=9), "mixed")
    try:
        before = fake.fake_conditional_nodes()
        if how == "round":
            b.step(1)
        elif how == "submit":
            b.submit(0, 1)
        else:
            info = xk.StepInfo()
            column(synth.small_column(L=9), "mixed", 0)._call("xk_step", 1e-8, ctypes.byref(info))
        assert fake.fake_conditional_nodes() == before
    finally:
        b.close()
        fake.fake_set_mps(0)


@pytest.mark.parametrize("S,small", [(40, True), (111, True), (112, True), (113, False), (161, False)])
def test_parcel_kernel_by_size(fake, column, S, small):
    """The parcel's kernel for systems in shared memory ends where its layout does."""
    p = synth.small_column(S=S, L=3, n_two=3 * S, n_three=3 * S // 4, n_photo=5, W=40, elements="chons" if S < 110 else "full")
    col = column(p, "fp64", 0)
    fake.fake_forget_launches()
    col._call("xk_parcel_begin", 100, 1e-8)
    assert (_launches_of(fake, "k_parcel_small")[0], _launches_of(fake, "k_parcel_iteration")[0]) == ((1, 0) if small else (0, 1))
    assert fake.fake_refused() == b""
