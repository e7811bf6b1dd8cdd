"""Resident kernels need all their blocks on the chip at once. Where that is refused the launches
they replaced serve the call, with the same results; where others use the GPU at the same time
(two handles on streams and threads of their own, a kernel that holds part of the SMs for longer
than a wait lasts) the call waits for its turn."""
import ctypes
import dataclasses
import functools
import shutil
import subprocess
import threading
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_08034_gb300 import _build
    _build.build()


@functools.lru_cache(maxsize=None)
def _case(dims=(36, 32, 40), u=0.01, s_in=0.4):
    from paper_2502_08034_gb300 import synth
    return synth.build_case("share%dx%dx%d" % dims, dims, 0.82, 4.0, 5, u, -0.10, s_in, 1e-10,
                            flow_device="cuda")


def _all(sv, case, precision):
    """Results of the calls that run resident, at check intervals of their own."""
    kw = dict(precision=precision, check_every=100)
    sv.reset_state()
    r = sv.solve(case.s_in, case.eta, 1e-10, **kw)
    s = sv.get_state()
    u, ru = sv.umt(1e-10, **kw)
    dm, db, ra = sv.adjoint("I_tot", 1e-10, **kw)
    return [np.array([r["I_tot"], r["sweeps"], u, ru["sweeps"], db, ra["sweeps"]]), s, dm]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_a_refused_launch_falls_back(precision):
    from paper_2502_08034_gb300 import rfb
    case, out = _case(), []
    for refused in (False, True):
        with rfb.Solver.from_case(case) as sv:
            before = sv.kernel_launches
            if refused:
                sv.selftest_refuse_resident()
            out.append(_all(sv, case, precision))
            launches = sv.kernel_launches - before
            assert (launches > 1000) == refused     # one a sweep, or one a cycle
            if precision == "mixed":
                assert (sv.tuned_fp32_kernel()[0] == "resident") != refused
            if refused:                             # a stream on which they are not refused
                sv.selftest_refuse_resident(False)
                sv.set_stream(torch.cuda.Stream())
                out.append(_all(sv, case, precision))
    for o in out[1:]:
        for x, y in zip(out[0], o):
            assert np.array_equal(x, y)


def test_a_refused_butler_volmer_solve_falls_back():
    """The parity bars of the resident and the streamed kernels."""
    from paper_2502_08034_gb300 import rfb
    case, out = dataclasses.replace(_case((13, 11, 15), 0.002, 0.2), k0=2e-5), []
    for refused in (False, True):
        with rfb.Solver.from_case(case) as sv:
            if refused:
                sv.selftest_refuse_resident()
            sv.solve(case.s_in, case.eta, 1e-12)
            r = sv.solve_bv(case.s_in, case.eta, 1e-30, start="sbv", max_sweeps=300, cycle=60,
                            allow_not_converged=True)
            out.append((r["I_tot"], sv.get_bv_state()))
    for k, bar in (("O", 1e-10), ("R", 1e-10), ("H", 1e-10), ("phi", 1e-7)):
        x, y = out[0][1][k], out[1][1][k]
        assert np.abs(x - y).max() <= bar * np.abs(y).max(), k
    assert out[0][0] == pytest.approx(out[1][0], rel=1e-9)


def test_two_handles_on_threads_of_their_own():
    from paper_2502_08034_gb300 import rfb
    case = _case((64, 64, 64))
    with rfb.Solver.from_case(case, stream=torch.cuda.Stream()) as a, \
            rfb.Solver.from_case(case, stream=torch.cuda.Stream()) as b:
        want = {p: _all(a, case, p) for p in ("fp64", "mixed")}
        got, errors = [], []

        def work(sv, precision):
            try:
                for _ in range(8):
                    got.append((precision, _all(sv, case, precision)))
            except Exception as e:                  # reported by the main thread
                errors.append(e)
        for pair in (("fp64", "fp64"), ("mixed", "fp64"), ("mixed", "mixed")):
            threads = [threading.Thread(target=work, args=(sv, p)) for sv, p in zip((a, b), pair)]
            for t in threads:
                t.start()
            for t in threads:
                t.join()
    assert not errors
    assert len(got) == 48
    for precision, o in got:
        for x, y in zip(want[precision], o):
            assert np.array_equal(x, y)


HOLD = r"""
#include <cuda_runtime.h>
// every block keeps its SM's shared memory for `ns` nanoseconds (an iteration limit besides)
__global__ void hold_kernel(unsigned long long ns, int* out) {
    extern __shared__ int s[];
    if (threadIdx.x) return;
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    int it = 0;
    do {
        __nanosleep(1000);
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    } while (t - t0 < ns && ++it < 10000000);
    s[0] = it;
    out[blockIdx.x] = s[0];
}
extern "C" int hold(int blocks, double seconds, void* stream, void* out) {
    const int smem = 200 * 1024;
    cudaFuncSetAttribute(hold_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    hold_kernel<<<blocks, 32, smem, (cudaStream_t)stream>>>((unsigned long long)(seconds * 1e9),
                                                            (int*)out);
    return (int)cudaGetLastError();
}
"""


def test_sms_held_by_another_stream_for_longer_than_a_wait(tmp_path):
    from paper_2502_08034_gb300 import rfb
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    (tmp_path / "hold.cu").write_text(HOLD)
    lib = str(tmp_path / "hold.so")
    subprocess.run([nvcc, "-gencode=arch=compute_103a,code=sm_103a", "-shared", "-Xcompiler",
                    "-fPIC", "-cudart", "shared", "-o", lib, str(tmp_path / "hold.cu")], check=True)
    hold = ctypes.CDLL(lib).hold
    hold.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p]
    other, out = torch.cuda.Stream(), torch.zeros(64, dtype=torch.int32, device="cuda")
    case = _case((64, 64, 64))
    with rfb.Solver.from_case(case, stream=torch.cuda.Stream()) as sv:
        for precision in ("mixed", "fp64"):
            want = _all(sv, case, precision)
            torch.cuda.synchronize()
            assert hold(40, 2.5, other.cuda_stream, out.data_ptr()) == 0
            time.sleep(0.05)
            got = _all(sv, case, precision)
            torch.cuda.synchronize()
            for x, y in zip(want, got):
                assert np.array_equal(x, y)
