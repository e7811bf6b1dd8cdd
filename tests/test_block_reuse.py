"""The batched double-float check walks its items in one block, reducing each through the same
shared memory. Its source is run here on host threads, one per lane, with the lanes that write a
block's result held back after the reduction's barrier: the sums of an item must not take part
of the next one's (an item of a lattice that has converged does nothing before its reduction)."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = r"""
#include <barrier>
#include <chrono>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <memory>
#include <thread>
#include <vector>
#define __device__
#define __global__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define __restrict__
#define __shared__ static
struct Dim { int x, y, z; };
constexpr int BX = 32, BY = 8, NRED = 8;
thread_local Dim threadIdx;
Dim blockIdx{0, 0, 0}, gridDim{1, 1, 1};
std::barrier<> block(BX * BY);
std::vector<std::unique_ptr<std::barrier<>>> warps;
double lanes[BX * BY];
int tid() { return threadIdx.y * BX + threadIdx.x; }
void __syncthreads() {
    block.arrive_and_wait();
    if (tid() < NRED) std::this_thread::sleep_for(std::chrono::milliseconds(20));
}
template <typename T, typename F> T over(T x, F f) {
    auto& w = *warps[tid() / 32];
    lanes[tid()] = (double)x;
    w.arrive_and_wait();
    const T r = f(lanes + tid() / 32 * 32);
    w.arrive_and_wait();
    return r;
}
unsigned __reduce_add_sync(unsigned, unsigned x) {
    return over(x, [](double* l) { double s = 0; for (int q = 0; q < 32; ++q) s += l[q]; return (unsigned)s; });
}
unsigned __reduce_max_sync(unsigned, unsigned x) {
    return over(x, [](double* l) { double s = 0; for (int q = 0; q < 32; ++q) s = std::fmax(s, l[q]); return (unsigned)s; });
}
double __shfl_xor_sync(unsigned, double x, int o) {
    return over(x, [o](double* l) { return l[(tid() & 31) ^ o]; });
}
unsigned __float_as_uint(float x) { unsigned u; std::memcpy(&u, &x, 4); return u; }
float __uint_as_float(unsigned u) { float x; std::memcpy(&x, &u, 4); return x; }
double widen(float x) { return x; }
using std::max;
struct Lattice { int nx; int64_t nxny; };
struct L2F {};
struct BatchInst { int active, cur; Lattice L; L2F K2; void* sdf[2]; void* delta[2]; void* r32; };
struct BatchItem { int inst, bx, kb, ke; };
template <bool FUSE, typename... P>
void check_df_column(const Lattice&, const L2F&, void*, void*, void*, void*, int, int, int, int kb,
                     int, float& sum2, float& vmax, int& bad) {
    sum2 += (float)kb;
    vmax = std::fmax(vmax, (float)kb);
    bad += 1;
}
"""
MAIN = r"""
int main() {
    for (int q = 0; q < 8; ++q) warps.push_back(std::make_unique<std::barrier<>>(32));
    BatchInst insts[2] = {};
    insts[0].active = 1;
    insts[0].L = insts[1].L = Lattice{32, 1024};
    // items of an active lattice (every cell adds kb) and of a converged one in turn
    BatchItem items[6];
    for (int q = 0; q < 6; ++q) items[q] = BatchItem{q & 1, 0, q + 1, q + 2};
    double partials[6 * NRED] = {};
    std::vector<std::thread> t;
    for (int y = 0; y < BY; ++y)
        for (int x = 0; x < BX; ++x)
            t.emplace_back([&, x, y] {
                threadIdx = Dim{x, y, 0};
                batch_check_df_kernel<true>(insts, items, 6, partials);
            });
    for (auto& q : t) q.join();
    for (int q = 0; q < 6; ++q)
        std::printf("%g %g %g\n", partials[q * NRED], partials[q * NRED + 6], partials[q * NRED + 7]);
}
"""


def _source():
    with open(os.path.join(ROOT, "paper_2502_08034_gb300", "csrc", "soc_kernels.cuh")) as f:
        text = f.read()
    out = []
    for start in (r"template <bool G>\n__device__ __forceinline__ void block_reduce_df\(",
                  r"template <bool FUSE>\n__global__ void [^{;]*?batch_check_df_kernel\("):
        at = re.search(start, text).start()
        out.append(text[at:text.index("\n}\n", at) + 3])
    return "\n".join(out)


def test_an_items_sums_do_not_mix_with_the_next_ones(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "reuse.cpp"
    src.write_text(HEAD + _source() + MAIN)
    exe = str(tmp_path / "reuse")
    subprocess.run([gxx, "-std=c++20", "-O1", "-pthread", "-w", "-o", exe, str(src)], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    got = [tuple(float(x) for x in line.split()) for line in out.splitlines()]
    assert got == [(1024.0 * (q + 1), 1024.0, q + 1.0) if q % 2 == 0 else (0.0, 0.0, 0.0)
                   for q in range(6)]
