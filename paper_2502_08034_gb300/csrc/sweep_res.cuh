// FP32 correction sweeps of a lattice that fits on the chip (local steps): one launch
// applies all the sweeps of a correction cycle.
//
// What bounds a small lattice is not its traffic but the fixed cost of a launch and the
// latency of one dependent round through L2 per sweep: one launch per sweep takes 6.1 us on
// every lattice from 16x16x32 to 92x92x100 (the rate at which the host can launch), of which a
// 64^3 lattice's traffic is 1.1 us. Here the lattice is cut into bricks of bx x by columns
// and CPT planes, one per CTA of a cooperative launch (all resident together). A thread owns
// a column of CPT cells and keeps their weights a_f, dt r and values in registers for the
// whole cycle; z neighbours are its own registers, x and y neighbours come from a
// double-buffered copy of the brick in shared memory. Only faces travel: after each sweep a
// CTA stores the new values of its faces into its neighbours' inboxes in global memory, each
// as one 64-bit word (value, sweep tag), and polls its own inbox for the words of that
// sweep. Value and tag arrive together (one 64-bit access), so a sweep costs one
// store-to-load latency and one block barrier instead of a launch, with no fence and no
// grid-wide barrier.
//
// The first warps own the brick's outer columns (the edge group). They alone wait for the side
// faces, behind a barrier of their own, and send theirs while the other warps work on the
// inside, which waits for its z words only after the cells that need none. So the time of a
// word on its way hides behind the inside: with one order for all warps 64^3 took 1.17 us a
// sweep, 75x61x118 1.90; now 0.94 and 1.62 (the smallest bricks, one warp, 0.78 and 0.82).
//
// Inboxes have two slots (sweep parity). A CTA overwrites the slot of sweep v with sweep
// v + 2 only after it computed v + 2, which needed the neighbour's words of v + 1, and the
// neighbour sends those after its edge group's barrier that follows its reads of v (the z faces
// pair thread with thread and need no barrier). Side faces go to the copy that the sweep
// reads, into places that the edge group alone uses. Tags grow from launch to launch (the
// handle keeps the count), so a slot is never cleared.
//
// Every update is dt_coef and dt_update with the operands and the order of the one-sweep
// kernel, so n sweeps here are bitwise n launches of sweep32d_kernel.
//
// Measured (us per sweep, 2000 a launch; launches before, resident now): 16x16x32 6.2 and
// 0.82, 64^3 6.2 and 0.94, 80x60x110 6.2 and 1.70, 88x88x108 6.4 and 2.41. About 0.75 us of it
// is the word latency (the smallest lattices); the rest is the shared-memory and issue time of
// a CTA's cells.
#pragma once

#include "sweep_dt.cuh"

namespace rfb {

constexpr int RES_T = 512;         // most threads of a CTA, columns of a brick (a launch has
                                   // the whole warps that its bricks need)
constexpr int RES_RING = 4;        // pairs of x / y halo words polled per edge thread, at most
// Shared memory of one plane of the brick: its rows without padding, one row below and one
// above (a warp's columns of one row never share a bank), then as much again for the columns left and right of the brick, each at its neighbour's index (the
// bank that its reader leaves free). With padded rows of bx + 2 every access of a warp that
// spans two rows took two turns: 528k cells 1.96 us a sweep. The pitch is fixed, so that a
// column's cells are immediate offsets and take no address registers.
constexpr int RES_ROWS = 640;      // bx * (by + 2) at most
constexpr int RES_PLANE = 2 * RES_ROWS;
// polls of one wait before it gives up (each a round trip to L2: about a second), unless the
// handle says otherwise
constexpr unsigned RES_SPIN_LIMIT = 1u << 20;

struct ResArgs {
    int nx, ny, nz;
    int bx, by;                    // columns of a brick (its planes: CPT)
    int gx, gy, gz;                // bricks
    int edge;                      // threads of the edge group (whole warps, the first ones)
    const float* __restrict__ u;   // FP32 face velocities * beta / h (low faces)
    const float* __restrict__ v;
    const float* __restrict__ w;   // nz + 1 planes
    const float* __restrict__ dt;  // per-cell step (0: not updated)
    const float* __restrict__ r;   // forcing
    const float* __restrict__ in;  // delta before the first sweep (nullptr: 0 everywhere)
    float* __restrict__ out;       // delta after the last sweep (another buffer than `in`)
    float omc, Dh;
    int n;                         // sweeps
    uint32_t tag;                  // the words of sweep v carry tag + v
    unsigned long long* inbox;     // CTAs x 2 slots x stride words
    int stride;
    unsigned int* err;             // set if a neighbour's word never arrives
    unsigned polls;                // of one wait, at most
};

// words of one inbox slot: the z faces, then the x and y faces
__host__ __device__ constexpr int res_stride(int cpt, int bx, int by) {
    return 2 * RES_T + 2 * cpt * (bx + by);
}
// From eight cells a column dt r is kept in shared memory (its own words only): the weights of
// eight cells and dt r spill at 128 registers a thread (80x60x110 1.77 us a sweep, without the
// spills 1.70; ten and twelve cells still spill 88 and 204 bytes).
__host__ __device__ constexpr bool res_dtr_shared(int cpt) { return cpt >= 8; }
// bytes of the two copies of a brick and its ring of neighbour columns, then dt r
__host__ __device__ constexpr int res_smem(int cpt) {
    return (2 * cpt * RES_PLANE + (res_dtr_shared(cpt) ? cpt * RES_T : 0)) * (int)sizeof(float);
}

__device__ __forceinline__ void res_send(unsigned long long* p, float x, uint32_t tag) {
    const unsigned long long word = ((unsigned long long)tag << 32) | __float_as_uint(x);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(word) : "memory");
}
// two words of a column's neighbouring cells (each 64-bit word by itself is whole)
__device__ __forceinline__ void res_send2(unsigned long long* p, float x, float y, uint32_t tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p),
                 "l"(t | __float_as_uint(x)), "l"(t | __float_as_uint(y))
                 : "memory");
}
__device__ __forceinline__ unsigned long long res_peek(const unsigned long long* p) {
    unsigned long long word;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(word) : "l"(p) : "memory");
    return word;
}

__device__ __forceinline__ void res_peek2(const unsigned long long* p,
                                          unsigned long long (&w)[2]) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
                 : "=l"(w[0]), "=l"(w[1])
                 : "l"(p)
                 : "memory");
}

// Column (x, y) of thread t in a brick of bx x by: the rows y = 0 and y = by - 1, then the rest of
// the columns x = 0 and x = bx - 1, then the inside.
__device__ __forceinline__ void res_column(int t, int bx, int by, int& x, int& y) {
    x = y = 0;
    if (t >= bx * by) return;                          // no column
    if (t < 2 * bx) {
        y = t < bx ? 0 : by - 1;
        x = t < bx ? t : t - bx;
        return;
    }
    t -= 2 * bx;
    if (t < 2 * (by - 2)) {
        y = 1 + (t >> 1);
        x = t & 1 ? bx - 1 : 0;
        return;
    }
    t -= 2 * (by - 2);
    y = 1 + t / (bx - 2);                              // bx > 2 here
    x = 1 + t % (bx - 2);
}
// barrier of the edge group alone (whole warps)
__device__ __forceinline__ void res_edge_sync(int threads) {
    asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}

template <int CPT, bool TR>   // CPT even
__global__ void __launch_bounds__(RES_T, 1) sweep32r_kernel(const ResArgs A) {
    extern __shared__ float res_s[];
    const int t = threadIdx.x;
    const int bx = A.bx, by = A.by;
    constexpr int plane = RES_PLANE, copy = CPT * RES_PLANE;
    const int b = blockIdx.x;
    const int ix = b % A.gx, iy = (b / A.gx) % A.gy, iz = b / (A.gx * A.gy);
    int x, y;
    res_column(t, bx, by, x, y);
    const bool mine = t < bx * by;                     // owns a column
    const bool edge = t < A.edge;                      // of the edge group (whole warps)
    const int i = ix * bx + x, j = iy * by + y, k0 = iz * CPT;
    for (int q = t; q < 2 * copy; q += (int)blockDim.x) res_s[q] = 0.f;

    // weights of the column (a cell outside the lattice has none: it stays 0)
    constexpr bool DTR_S = res_dtr_shared(CPT);
    CoefD kc[CPT];
    float dtr[DTR_S ? 1 : CPT], d[CPT];
    float* const dtr_s = res_s + 2 * copy + t;
    const int64_t nxny = (int64_t)A.nx * A.ny;
    const int64_t c0 = i + (int64_t)A.nx * j + nxny * k0;
    const bool in_xy = mine && i < A.nx && j < A.ny;
#pragma unroll
    for (int e = 0; e < CPT; ++e) {
        const bool in = in_xy && k0 + e < A.nz;
        const int64_t c = c0 + nxny * e;
        const float dt = in ? __ldg(A.dt + c) : 0.f;
        const float uL = in ? __ldg(A.u + c) : 0.f;
        const float uH = in && i + 1 < A.nx ? __ldg(A.u + c + 1) : 0.f;
        const float vL = in ? __ldg(A.v + c) : 0.f;
        const float vH = in && j + 1 < A.ny ? __ldg(A.v + c + A.nx) : 0.f;
        const float wL = in ? __ldg(A.w + c) : 0.f;
        const float wH = in ? __ldg(A.w + c + nxny) : 0.f;
        kc[e] = dt_coef<TR>(dt, A.Dh, uL, uH, vL, vH, wL, wH);
        const float f = dt * (in ? __ldg(A.r + c) : 0.f);
        if (DTR_S) dtr_s[e * RES_T] = f;
        else dtr[DTR_S ? 0 : e] = f;
        d[e] = in && A.in ? __ldg(A.in + c) : 0.f;
    }

    // halo words of this thread: the two z faces of its column (bits 0 and 1 of `want`, set
    // where there is a neighbour) and, in the edge group, up to RES_RING pairs of the x and y
    // faces (bits 2, ..)
    const int nfx = CPT * by, nfy = CPT * bx;          // words of one x face, one y face (a
                                                       // column's CPT words together)
    uint32_t want = 0;
    if (mine && iz > 0) want |= 1u;
    if (mine && iz + 1 < A.gz) want |= 2u;
    uint32_t dst[RES_RING / 2] = {};                   // two 16-bit indices each
#pragma unroll
    for (int m = 0; m < RES_RING; ++m) {
        int q = 2 * (t + m * A.edge);
        if (!edge || q >= 2 * (nfx + nfy)) continue;
        int at;
        if (q < 2 * nfx) {
            const bool hi = q >= nfx;
            if (hi) q -= nfx;
            at = (q % CPT) * plane + RES_ROWS + (q / CPT + 1) * bx + (hi ? bx : -1);
            if (hi ? ix + 1 < A.gx : ix > 0) want |= 4u << m;
        } else {
            q -= 2 * nfx;
            const bool hi = q >= nfy;
            if (hi) q -= nfy;
            at = (q % CPT) * plane + (hi ? by + 1 : 0) * bx + q / CPT;
            if (hi ? iy + 1 < A.gy : iy > 0) want |= 4u << m;
        }
        dst[m / 2] |= (uint32_t)at << 16 * (m & 1);
    }
    // words this column sends to, from slot 0 (-1: no neighbour there; a brick is at least
    // two columns wide each way, so a column is on one x face and one y face at most)
    auto box = [&](int c) { return c * 2 * A.stride; };
    const int own = box(b);
    int to_zm = -1, to_zp = -1, to_x = -1, to_y = -1;
    if (mine) {
        if (iz > 0) to_zm = box(b - A.gx * A.gy) + RES_T + t;
        if (iz + 1 < A.gz) to_zp = box(b + A.gx * A.gy) + t;
        if (x == 0 && ix > 0) to_x = box(b - 1) + 2 * RES_T + nfx + y * CPT;
        if (x == bx - 1 && ix + 1 < A.gx) to_x = box(b + 1) + 2 * RES_T + y * CPT;
        if (y == 0 && iy > 0) to_y = box(b - A.gx) + 2 * RES_T + 2 * nfx + nfy + x * CPT;
        if (y == by - 1 && iy + 1 < A.gy) to_y = box(b + A.gx) + 2 * RES_T + 2 * nfx + x * CPT;
    }
    const int o = bx + y * bx + x;                     // this column in a plane, its x neighbours
    const int oxm = x == 0 ? RES_ROWS + o - 1 : o - 1;
    const int oxp = x == bx - 1 ? RES_ROWS + o + 1 : o + 1;
    float zlo = 0.f, zhi = 0.f;                        // values below and above the column
    bool good = true;
    __syncthreads();
    if (A.in) {                                        // the brick and its ring before sweep 1
        if (in_xy && k0 > 0) zlo = __ldg(A.in + c0 - nxny);
        if (in_xy && k0 + CPT < A.nz) zhi = __ldg(A.in + c0 + nxny * CPT);
        for (int q = t; q < copy; q += (int)blockDim.x) {
            // row yy of the brick (0: the row below it); the second half of a plane holds the
            // columns left (index -1 of row yy) and right (index bx) of the brick
            const int e = q / plane, p = q % plane, r = p % RES_ROWS;
            int yy = r / bx, xx = r % bx;
            if (p >= RES_ROWS) {
                if (xx == bx - 1) { ++yy; xx = -1; }
                else if (xx == 0) { --yy; xx = bx; }
                else continue;
                if (yy < 1 || yy > by) continue;
            }
            const int gi = ix * bx + xx, gj = iy * by + yy - 1, gk = k0 + e;
            if (yy < by + 2 && gi >= 0 && gi < A.nx && gj >= 0 && gj < A.ny && gk < A.nz)
                res_s[q] = __ldg(A.in + gi + (int64_t)A.nx * gj + nxny * gk);
        }
        __syncthreads();
    }
    // the words of sweep ver - 1 this thread waits for (of `which`): z values into zlo and zhi,
    // side faces into the brick's copy; a warp stays together until all its lanes have theirs
    auto take = [&](int ver, uint32_t which, float* Sr) {
        const uint32_t tag = A.tag + (uint32_t)(ver - 1);
        const unsigned long long* in = A.inbox + ((ver - 1) & 1) * A.stride + own;
        uint32_t pend = good ? want & which : 0u;
        for (unsigned spin = 0; __any_sync(0xffffffffu, pend != 0u); ++spin) {
            unsigned long long zw[2], word[RES_RING][2];
#pragma unroll
            for (int m = 0; m < 2; ++m)
                if (pend & (1u << m)) zw[m] = res_peek(in + t + m * RES_T);
#pragma unroll
            for (int m = 0; m < RES_RING; ++m)
                if (pend & (4u << m)) res_peek2(in + 2 * RES_T + 2 * (t + m * A.edge), word[m]);
            if ((pend & 1u) && (uint32_t)(zw[0] >> 32) == tag) {
                zlo = __uint_as_float((uint32_t)zw[0]);
                pend &= ~1u;
            }
            if ((pend & 2u) && (uint32_t)(zw[1] >> 32) == tag) {
                zhi = __uint_as_float((uint32_t)zw[1]);
                pend &= ~2u;
            }
#pragma unroll
            for (int m = 0; m < RES_RING; ++m)
                if ((pend & (4u << m)) && (uint32_t)(word[m][0] >> 32) == tag &&
                    (uint32_t)(word[m][1] >> 32) == tag) {
                    const uint32_t at = dst[m / 2] >> 16 * (m & 1) & 0xffffu;
                    Sr[at] = __uint_as_float((uint32_t)word[m][0]);
                    Sr[at + plane] = __uint_as_float((uint32_t)word[m][1]);
                    pend &= ~(4u << m);
                }
            if (spin + 1 >= A.polls && pend) {         // give up, and wait no more
                atomicExch(A.err, 1u);
                good = false;
                pend = 0;
            }
        }
    };
    for (int ver = 1; ver <= A.n; ++ver) {
        float* Sr = res_s + ((ver - 1) & 1) * copy;             // the brick before this sweep
        float* Sw = res_s + (ver & 1) * copy + o;               // and after
        const uint32_t tag = A.tag + (uint32_t)ver;
        unsigned long long* const slot = A.inbox + (ver & 1) * A.stride;
        const bool more = ver < A.n;
        if (edge && ver > 1) {
            take(ver, ~0u, Sr);
            res_edge_sync(A.edge);                     // other threads' side words
        }
        auto update = [&](int e, float zm, float zp) {
            const int q = e * plane;
            return dt_update(kc[e], A.omc, d[e], DTR_S ? dtr_s[e * RES_T] : dtr[DTR_S ? 0 : e],
                             Sr[q + oxm], Sr[q + oxp], Sr[q + o - bx], Sr[q + o + bx], zm, zp);
        };
        // the inside of the column, then (its z words may have come meanwhile) its ends
        const float second = d[1], second_last = d[CPT - 2];
        float prev = d[0];
#pragma unroll
        for (int e = 1; e < CPT - 1; ++e) {
            const float val = update(e, prev, d[e + 1]);
            prev = d[e];
            d[e] = val;
        }
        if (!edge && ver > 1) take(ver, 3u, Sr);
        const float lo = update(0, zlo, second), hi = update(CPT - 1, second_last, zhi);
        d[0] = lo;
        d[CPT - 1] = hi;
        if (more) {
            if (to_zm >= 0) res_send(slot + to_zm, lo, tag);
            if (to_zp >= 0) res_send(slot + to_zp, hi, tag);
            if (edge) {
                if (to_x >= 0) {
#pragma unroll
                    for (int e = 0; e < CPT; e += 2) res_send2(slot + to_x + e, d[e], d[e + 1], tag);
                }
                if (to_y >= 0) {
#pragma unroll
                    for (int e = 0; e < CPT; e += 2) res_send2(slot + to_y + e, d[e], d[e + 1], tag);
                }
            }
            if (mine) {
#pragma unroll
                for (int e = 0; e < CPT; ++e) Sw[e * plane] = d[e];
            }
            __syncthreads();
        }
    }
    if (in_xy) {
#pragma unroll
        for (int e = 0; e < CPT; ++e)
            if (k0 + e < A.nz) A.out[c0 + nxny * e] = d[e];
    }
}

// ---------------------------------------------------------------------------------
// Resident FP64 sweeps with the assembled operator, s <- s + dt RHS(s) (ADJ: the transposed
// step lam <- lam + dt (L^T lam + g)). The scheme of the FP32 kernel: bricks, columns of CPT
// cells per thread, faces as tagged words, here two 64-bit words a value (its halves). What
// bounds it is the FP64 pipe: 8 DFMA a cell at 2 lanes a clock and SM, 2.9 us for 48x48x96,
// so the whole warps a cut takes decide its time and shared memory costs nothing beside it.
// Operands and order are those of sweep64c_kernel and adjoint64c_kernel: bitwise the same.
//
// Measured (us per sweep, launches before and resident now): 16x16x32 8.2 and 1.6, 48^3 8.2 and
// 2.3, 48x48x96 10.3 and 3.7, 64^3 10.2 and 4.6, 60x60x110 12.3 and 6.5 (one order for all warps,
// as above: 1.5, 2.5, 4.6, 5.6, 7.9).
// ---------------------------------------------------------------------------------
constexpr int RES64_RING = 4;      // x / y halo values polled per edge thread, at most
// coefficients of a cell kept in shared memory (the last ones; registers hold the others):
// eight doubles for three to six cells do not fit beside the values at 128 registers (four
// cells: 264 bytes of spills with none of them in shared memory, 40 with two a cell; 64^3 4.7
// and 4.5 us a sweep)
__host__ __device__ constexpr int res64_shared(int cpt) { return cpt >= 6 ? 4 : cpt >= 5 ? 3 : cpt >= 4 ? 2 : cpt >= 3 ? 1 : 0; }
__host__ __device__ constexpr int res64_smem(int cpt) {
    return (2 * cpt * RES_PLANE + cpt * res64_shared(cpt) * RES_T) * (int)sizeof(double);
}
// 16-byte entries of one inbox slot
__host__ __device__ constexpr int res64_stride(int cpt, int bx, int by) {
    return 2 * RES_T + 2 * cpt * (bx + by);
}

struct Res64Args {
    Lattice L;
    int bx, by, gx, gy, gz, edge;  // as in ResArgs
    L64 K;
    const float* __restrict__ dtc; // per-cell step, nullptr: dt
    double dt;
    const double* __restrict__ in; // before the first sweep
    double* __restrict__ out;      // after the last (another buffer)
    const double* __restrict__ g;  // ADJ: the source
    int umt, n;
    uint32_t tag;
    unsigned long long* inbox;     // CTAs x 2 slots x stride entries of two words
    int stride;
    unsigned int* err;
    unsigned polls;
};

__device__ __forceinline__ void res_send64(unsigned long long* p, double x, uint32_t tag) {
    const unsigned long long t = (unsigned long long)tag << 32, v = __double_as_longlong(x);
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p),
                 "l"(t | (v & 0xffffffffull)), "l"(t | (v >> 32))
                 : "memory");
}
__device__ __forceinline__ bool res_take64(const unsigned long long (&w)[2], uint32_t tag,
                                           double* x) {
    if ((uint32_t)(w[0] >> 32) != tag || (uint32_t)(w[1] >> 32) != tag) return false;
    *x = __longlong_as_double((long long)((w[0] & 0xffffffffull) | (w[1] << 32)));
    return true;
}

template <int CPT, bool ADJ>   // CPT >= 2
__global__ void __launch_bounds__(RES_T, 1) sweep64r_kernel(const Res64Args A) {
    extern __shared__ double res_s64[];
    constexpr int plane = RES_PLANE, copy = CPT * RES_PLANE;
    constexpr int NS = res64_shared(CPT), NR = 8 - NS;
    const int t = threadIdx.x;
    const int nx = A.L.nx, ny = A.L.ny, nz = A.L.nz;
    const int bx = A.bx, by = A.by;
    const int b = blockIdx.x;
    const int ix = b % A.gx, iy = (b / A.gx) % A.gy, iz = b / (A.gx * A.gy);
    int x, y;
    res_column(t, bx, by, x, y);
    const bool edge = t < A.edge;
    const int i = ix * bx + x, j = iy * by + y, k0 = iz * CPT;
    const int64_t nxny = A.L.nxny, N = nxny * nz;
    const int64_t c0 = i + (int64_t)nx * j + nxny * k0;
    const bool mine = t < bx * by;
    const bool in_xy = mine && i < nx && j < ny;

    // coefficients in the order of use: diagonal, source, then the six neighbours
    double kr[CPT][NR], d[CPT], dt[CPT];
    double* const ks = res_s64 + 2 * copy + t;
    uint32_t upd = 0;
#pragma unroll
    for (int e = 0; e < CPT; ++e) {
        const bool in = in_xy && k0 + e < nz;
        const int64_t c = c0 + nxny * e;
        const unsigned f = in ? A.L.flags[c] : 0u;
        const bool u = (f & F_FLUID) && !(A.umt && (f & F_ELEC));
        if (u) upd |= 1u << e;
        double q[8];
        q[0] = u ? A.K.diag[c] : 0.0;
        if (ADJ) {   // from each neighbour's row the coefficient that points back here
            q[1] = u ? A.g[c] : 0.0;
            q[2] = u && i > 0 ? A.K.f[1][c - 1] : 0.0;
            q[3] = u && i + 1 < nx ? A.K.f[0][c + 1] : 0.0;
            q[4] = u && j > 0 ? A.K.f[3][c - nx] : 0.0;
            q[5] = u && j + 1 < ny ? A.K.f[2][c + nx] : 0.0;
            q[6] = u && c >= nxny ? A.K.f[5][c - nxny] : 0.0;
            q[7] = u && c + nxny < N ? A.K.f[4][c + nxny] : 0.0;
        } else {
            q[1] = u ? A.K.b[c] : 0.0;
#pragma unroll
            for (int m = 0; m < 6; ++m) q[2 + m] = u ? A.K.f[m][c] : 0.0;
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            if (m < NR) kr[e][m < NR ? m : 0] = q[m];
            else ks[(e * NS + m - NR) * RES_T] = q[m];
        }
        dt[e] = u ? (A.dtc ? (double)A.dtc[c] : A.dt) : 0.0;
        d[e] = in ? A.in[c] : 0.0;
    }
    // the brick and the columns around it before the first sweep (0 outside the lattice)
    for (int q = t; q < 2 * copy; q += (int)blockDim.x) {
        const int e = q % copy / plane, p = q % plane, r = p % RES_ROWS;
        int yy = r / bx, xx = r % bx;
        bool at = q < copy;
        if (p >= RES_ROWS) {
            if (xx == bx - 1) { ++yy; xx = -1; }
            else if (xx == 0) { --yy; xx = bx; }
            else at = false;
            if (yy < 1 || yy > by) at = false;
        }
        const int gi = ix * bx + xx, gj = iy * by + yy - 1, gk = k0 + e;
        at = at && yy < by + 2 && gi >= 0 && gi < nx && gj >= 0 && gj < ny && gk < nz;
        res_s64[q] = at ? A.in[gi + (int64_t)nx * gj + nxny * gk] : 0.0;
    }
    double zlo = in_xy && k0 > 0 ? A.in[c0 - nxny] : 0.0;
    double zhi = in_xy && k0 + CPT < nz ? A.in[c0 + nxny * CPT] : 0.0;

    const int nfx = CPT * by, nfy = CPT * bx;
    uint32_t want = 0;
    if (mine && iz > 0) want |= 1u;
    if (mine && iz + 1 < A.gz) want |= 2u;
    uint32_t dst[RES64_RING / 2] = {};                   // two 16-bit indices each
#pragma unroll
    for (int m = 0; m < RES64_RING; ++m) {
        int q = t + m * A.edge;
        if (!edge || q >= 2 * (nfx + nfy)) continue;
        int at;
        if (q < 2 * nfx) {
            const bool hi = q >= nfx;
            if (hi) q -= nfx;
            at = (q % CPT) * plane + RES_ROWS + (q / CPT + 1) * bx + (hi ? bx : -1);
            if (hi ? ix + 1 < A.gx : ix > 0) want |= 4u << m;
        } else {
            q -= 2 * nfx;
            const bool hi = q >= nfy;
            if (hi) q -= nfy;
            at = (q % CPT) * plane + (hi ? by + 1 : 0) * bx + q / CPT;
            if (hi ? iy + 1 < A.gy : iy > 0) want |= 4u << m;
        }
        dst[m / 2] |= (uint32_t)at << 16 * (m & 1);
    }
    auto box = [&](int c) { return c * 2 * A.stride; };
    const int own = box(b);
    int to_zm = -1, to_zp = -1, to_x = -1, to_y = -1;
    if (mine) {
        if (iz > 0) to_zm = box(b - A.gx * A.gy) + RES_T + t;
        if (iz + 1 < A.gz) to_zp = box(b + A.gx * A.gy) + t;
        if (x == 0 && ix > 0) to_x = box(b - 1) + 2 * RES_T + nfx + y * CPT;
        if (x == bx - 1 && ix + 1 < A.gx) to_x = box(b + 1) + 2 * RES_T + y * CPT;
        if (y == 0 && iy > 0) to_y = box(b - A.gx) + 2 * RES_T + 2 * nfx + nfy + x * CPT;
        if (y == by - 1 && iy + 1 < A.gy) to_y = box(b + A.gx) + 2 * RES_T + 2 * nfx + x * CPT;
    }
    const int o = bx + y * bx + x;
    const int oxm = x == 0 ? RES_ROWS + o - 1 : o - 1;
    const int oxp = x == bx - 1 ? RES_ROWS + o + 1 : o + 1;
    bool good = true;
    __syncthreads();
    auto take = [&](int ver, uint32_t which, double* Sr) {
        const uint32_t tag = A.tag + (uint32_t)(ver - 1);
        const unsigned long long* in = A.inbox + 2 * (((ver - 1) & 1) * A.stride + own);
        uint32_t pend = good ? want & which : 0u;
        for (unsigned spin = 0; __any_sync(0xffffffffu, pend != 0u); ++spin) {
            unsigned long long word[2 + RES64_RING][2];
#pragma unroll
            for (int m = 0; m < 2 + RES64_RING; ++m)
                if (pend & (1u << m))
                    res_peek2(in + 2 * (m < 2 ? t + m * RES_T : 2 * RES_T + t + (m - 2) * A.edge),
                              word[m]);
#pragma unroll
            for (int m = 0; m < 2 + RES64_RING; ++m) {
                double val;
                if ((pend & (1u << m)) && res_take64(word[m], tag, &val)) {
                    if (m == 0) zlo = val;
                    else if (m == 1) zhi = val;
                    else Sr[dst[m >= 2 ? (m - 2) / 2 : 0] >> 16 * (m & 1) & 0xffffu] = val;
                    pend &= ~(1u << m);
                }
            }
            if (spin + 1 >= A.polls && pend) {
                atomicExch(A.err, 1u);
                good = false;
                pend = 0;
            }
        }
    };
    for (int ver = 1; ver <= A.n; ++ver) {
        double* Sr = res_s64 + ((ver - 1) & 1) * copy;
        double* Sw = res_s64 + (ver & 1) * copy + o;
        const uint32_t tag = A.tag + (uint32_t)ver;
        unsigned long long* const slot = A.inbox + 2 * ((ver & 1) * A.stride);
        const bool more = ver < A.n;
        if (edge && ver > 1) {
            take(ver, ~0u, Sr);
            res_edge_sync(A.edge);
        }
        auto coef = [&](int e, int m) {
            return m < NR ? kr[e][m < NR ? m : 0] : ks[(e * NS + m - NR) * RES_T];
        };
        auto update = [&](int e, double zm, double zp) {
            const double* P = Sr + e * plane;
            double r = fma(coef(e, 0), d[e], coef(e, 1));
            r = fma(coef(e, 2), P[oxm], r);
            r = fma(coef(e, 3), P[oxp], r);
            r = fma(coef(e, 4), P[o - bx], r);
            r = fma(coef(e, 5), P[o + bx], r);
            r = fma(coef(e, 6), zm, r);
            r = fma(coef(e, 7), zp, r);
            const double val = fma(dt[e], r, d[e]);
            return (upd >> e) & 1u ? val : d[e];
        };
        const bool work = (t & ~31) < bx * by;         // a warp without columns does no FP64
        const double second = d[1], second_last = d[CPT - 2];
        if (work) {
            double prev = d[0];
#pragma unroll
            for (int e = 1; e < CPT - 1; ++e) {
                const double val = update(e, prev, d[e + 1]);
                prev = d[e];
                d[e] = val;
            }
        }
        if (!edge && ver > 1) take(ver, 3u, Sr);
        if (work) {
            const double lo = update(0, zlo, second), hi = update(CPT - 1, second_last, zhi);
            d[0] = lo;
            d[CPT - 1] = hi;
        }
        if (more) {
            if (to_zm >= 0) res_send64(slot + 2 * to_zm, d[0], tag);
            if (to_zp >= 0) res_send64(slot + 2 * to_zp, d[CPT - 1], tag);
            if (edge) {
                if (to_x >= 0) {
#pragma unroll
                    for (int e = 0; e < CPT; ++e) res_send64(slot + 2 * (to_x + e), d[e], tag);
                }
                if (to_y >= 0) {
#pragma unroll
                    for (int e = 0; e < CPT; ++e) res_send64(slot + 2 * (to_y + e), d[e], tag);
                }
            }
            if (mine) {
#pragma unroll
                for (int e = 0; e < CPT; ++e) Sw[e * plane] = d[e];
            }
            __syncthreads();
        }
    }
    if (in_xy) {
#pragma unroll
        for (int e = 0; e < CPT; ++e)
            if (k0 + e < nz) A.out[c0 + nxny * e] = d[e];
    }
}

}  // namespace rfb
