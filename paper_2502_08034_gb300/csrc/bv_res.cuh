// Butler-Volmer model on a lattice that fits on the chip: the potential solve and the species
// sweeps of a cycle as one launch each (the scheme and the tagged words of sweep_res.cuh).
//
// A small lattice's potential solve was six launches per conjugate-gradient iteration, about
// 50 us whatever its size, with a host wait every 50 iterations; its species sweeps were one
// launch each and recomputed two exponentials, three divisions and every migration term per
// cell, although the potential is fixed between solves. Here
//   - bv_cgr_kernel runs a whole potential solve: face conductivities and vectors in registers,
//     two reductions over all CTAs per iteration, the stopping rule on the device;
//   - bv_sweepr_kernel forms each cell's coefficients once per launch (the right-hand side of
//     a species is linear in the concentrations at a fixed potential) and then sweeps.
//
// Measured on 20x14x26 (from the SBV state to residual 1e-8: 6500 sweeps, 14200 iterations):
// 775 ms before, 155 ms now; an iteration 50 us before and 7.7 now, most of it the latency of
// dependent FP64 operations (64 clocks a warp each) in the two reductions.
#pragma once

#include "bv_kernels.cuh"
#include "sweep_res.cuh"

namespace rfb {

struct ResCut {                    // bricks of a lattice (see ResArgs)
    int bx, by, gx, gy, gz;
};

// A thread's column of CPT cells in its brick, the 16-byte inbox entries it sends to and polls
// (offsets from slot 0 of the first inbox; an inbox slot holds NV values per face cell, one
// sub-slot of `stride` entries after the other), and its places in the shared copy (value v of
// the brick's cells after CPT planes of each value before it).
template <int CPT, int RING, int NV>
struct ResBrick {
    bool mine;                     // owns a column
    int i, j, k0;
    int o, oxm, oxp, bx;
    int own, to_zm, to_zp, to_x, to_y;
    int src[RING], dst[RING];      // polled x and y face words, their shared-memory places
    uint32_t want;                 // bits 0, 1: z faces; 2 ..: src

    __device__ __forceinline__ void init(const ResCut& c, int stride) {
        const int t = threadIdx.x, b = blockIdx.x;
        const int ix = b % c.gx, iy = (b / c.gx) % c.gy, iz = b / (c.gx * c.gy);
        const int x = t % c.bx, y = t / c.bx;
        bx = c.bx;
        mine = y < c.by;
        i = ix * bx + x;
        j = iy * c.by + y;
        k0 = iz * CPT;
        o = bx + t;
        oxm = x == 0 ? RES_ROWS + o - 1 : o - 1;
        oxp = x == bx - 1 ? RES_ROWS + o + 1 : o + 1;
        const int nfx = CPT * c.by, nfy = CPT * bx, nr = 2 * (nfx + nfy);
        want = 0;
        if (mine && iz > 0) want |= 1u;
        if (mine && iz + 1 < c.gz) want |= 2u;
#pragma unroll
        for (int m = 0; m < RING; ++m) {
            int q = t + m * (int)blockDim.x;
            src[m] = dst[m] = 0;
            if (q >= NV * nr) continue;
            const int v = q / nr;
            q -= v * nr;
            src[m] = v * stride + 2 * RES_T + q;
            dst[m] = v * CPT * RES_PLANE;
            if (q < 2 * nfx) {
                const bool hi = q >= nfx;
                if (hi) q -= nfx;
                dst[m] += (q % CPT) * RES_PLANE + RES_ROWS + (q / CPT + 1) * bx + (hi ? bx : -1);
                if (hi ? ix + 1 < c.gx : ix > 0) want |= 4u << m;
            } else {
                q -= 2 * nfx;
                const bool hi = q >= nfy;
                if (hi) q -= nfy;
                dst[m] += (q % CPT) * RES_PLANE + (hi ? c.by + 1 : 0) * bx + q / CPT;
                if (hi ? iy + 1 < c.gy : iy > 0) want |= 4u << m;
            }
        }
        auto box = [&](int q) { return q * 2 * NV * stride; };
        own = box(b);
        to_zm = to_zp = to_x = to_y = -1;
        if (mine) {
            if (iz > 0) to_zm = box(b - c.gx * c.gy) + RES_T + t;
            if (iz + 1 < c.gz) to_zp = box(b + c.gx * c.gy) + t;
            if (x == 0 && ix > 0) to_x = box(b - 1) + 2 * RES_T + nfx + y * CPT;
            if (x == bx - 1 && ix + 1 < c.gx) to_x = box(b + 1) + 2 * RES_T + y * CPT;
            if (y == 0 && iy > 0) to_y = box(b - c.gx) + 2 * RES_T + 2 * nfx + nfy + x * CPT;
            if (y == c.by - 1 && iy + 1 < c.gy) to_y = box(b + c.gx) + 2 * RES_T + 2 * nfx + x * CPT;
        }
    }
    // the column's values val[0 .. CPT-1] to the neighbours they touch; slot: the words of this
    // exchange's slot and sub-slot
    __device__ __forceinline__ void send(unsigned long long* slot, const double (&val)[CPT],
                                         uint32_t tag) const {
        if (to_zm >= 0) res_send64(slot + 2 * to_zm, val[0], tag);
        if (to_zp >= 0) res_send64(slot + 2 * to_zp, val[CPT - 1], tag);
        if (to_x >= 0) {
#pragma unroll
            for (int e = 0; e < CPT; ++e) res_send64(slot + 2 * (to_x + e), val[e], tag);
        }
        if (to_y >= 0) {
#pragma unroll
            for (int e = 0; e < CPT; ++e) res_send64(slot + 2 * (to_y + e), val[e], tag);
        }
    }
    // the neighbours' words of this exchange: the values below and above the column into
    // zlo, zhi, the side faces' into ring (left alone where there is no neighbour). `good`
    // turns false when a word did not come within the limit (err is set, what came is kept)
    // and must have been the thread's own from the start; called by whole warps, which stay
    // together until every lane has its words.
    __device__ __forceinline__ void poll(const unsigned long long* slot, int stride, uint32_t tag,
                                         double (&zlo)[NV], double (&zhi)[NV],
                                         double (&ring)[RING], unsigned int* err,
                                         unsigned polls, bool& good) const {
        constexpr int NZ = 2 * NV, NI = NZ + RING;     // z words of value v: bits 2 v, 2 v + 1
        const unsigned long long* in = slot + 2 * own;
        uint32_t pend = (want >> 2) << NZ;
#pragma unroll
        for (int v = 0; v < NV; ++v) pend |= (want & 3u) << (2 * v);
        if (!good) pend = 0;
        for (unsigned spin = 0; __any_sync(0xffffffffu, pend != 0u); ++spin) {
            unsigned long long word[NI][2];
#pragma unroll
            for (int m = 0; m < NI; ++m)
                if (pend & (1u << m))
                    res_peek2(in + 2 * (m < NZ ? (m >> 1) * stride + (m & 1) * RES_T +
                                                     (int)threadIdx.x
                                               : src[m >= NZ ? m - NZ : 0]),
                              word[m]);
#pragma unroll
            for (int m = 0; m < NI; ++m) {
                double val;
                if ((pend & (1u << m)) && res_take64(word[m], tag, &val)) {
                    if (m >= NZ) ring[m >= NZ ? m - NZ : 0] = val;
                    else if (m & 1) zhi[m < NZ ? m >> 1 : 0] = val;
                    else zlo[m < NZ ? m >> 1 : 0] = val;
                    pend &= ~(1u << m);
                }
            }
            if (spin + 1 >= polls && pend) {
                atomicExch(err, 1u);
                good = false;
                pend = 0;
            }
        }
    }
};

// A reduction over every CTA of the launch: each leaves its block's value, tagged, in its
// place of one row; the first warp of each CTA reads the row and reduces it in the same order
// (the result is the same bits everywhere), then the block takes it from shared memory. Two
// rows in turn: a CTA writes reduction k + 2 after it read k + 1, which every CTA wrote after
// it had read k. Only the first warp adds across warps and CTAs, and forms what follows from
// the sum (`post`): on the narrow FP64 pipe sixteen warps doing the same tree and the same
// division took 20 us an iteration.
constexpr int RES_LANE = 5;        // places a lane reads: at most 160 CTAs
struct ResReduce {
    unsigned long long* rows;      // 2 rows of CTAs entries (16 bytes)
    double* sh;                    // 32 + 2 doubles of shared memory
    uint32_t tag;                  // of the next reduction
    unsigned int* err;
    unsigned polls;                // of one wait, at most
    bool good;                     // this thread may wait (none of its waits gave up)
    bool dead;                     // a wait of this CTA gave up (the same in all its threads)

    template <typename Op>
    __device__ __forceinline__ double warp(double x, Op op) {
        for (int o = 16; o > 0; o >>= 1) x = op(x, __shfl_xor_sync(0xffffffffu, x, o));
        return x;
    }
    // op commutative, none: its neutral value; the result, and post(result)
    template <typename Op, typename Post>
    __device__ __forceinline__ double2 all(double x, double none, Op op, Post post) {
        const int t = threadIdx.x, lane = t & 31, w = t >> 5;
        const int n = gridDim.x;
        x = warp(x, op);
        if (lane == 0) sh[w] = x;
        if (__syncthreads_or(!good)) { good = false; dead = true; }
        if (w == 0) {
            unsigned long long* row = rows + 2 * (tag & 1u) * n;
            x = lane < (int)(blockDim.x >> 5) ? sh[lane] : none;
            if (blockDim.x > 32) x = warp(x, op);
            if (lane == 0) res_send64(row + 2 * blockIdx.x, x, tag);
            __syncwarp();              // sent before any lane of this warp starts polling
            double v[RES_LANE];
            uint32_t pend = 0;
#pragma unroll
            for (int m = 0; m < RES_LANE; ++m) {
                v[m] = none;
                if (good && lane + 32 * m < n) pend |= 1u << m;
            }
            for (unsigned spin = 0; __any_sync(0xffffffffu, pend != 0u); ++spin) {
                unsigned long long word[RES_LANE][2];
#pragma unroll
                for (int m = 0; m < RES_LANE; ++m)
                    if (pend & (1u << m)) res_peek2(row + 2 * (lane + 32 * m), word[m]);
#pragma unroll
                for (int m = 0; m < RES_LANE; ++m)
                    if ((pend & (1u << m)) && res_take64(word[m], tag, &v[m])) pend &= ~(1u << m);
                if (spin + 1 >= polls && pend) {
                    atomicExch(err, 1u);
                    good = false;
                    pend = 0;
                }
            }
            double sum = v[0];
#pragma unroll
            for (int m = 1; m < RES_LANE; ++m) sum = op(sum, v[m]);
            sum = warp(sum, op);
            if (lane == 0) {
                sh[32] = sum;
                sh[33] = post(sum);
            }
        }
        __syncthreads();
        ++tag;
        return make_double2(sh[32], sh[33]);
    }
    template <typename Op>
    __device__ __forceinline__ double all(double x, double none, Op op) {
        return all(x, none, op, [](double v) { return v; }).x;
    }
};

struct BVCgArgs {
    BVArgs B;
    ResCut cut;
    const double* __restrict__ kcell;
    const double* __restrict__ kmem;
    const double* __restrict__ bphi;
    double* phi;                   // in: start, out: solution
    double tol;                    // done when max |residual| <= tol (or at the rounding floor)
    int max_it;
    uint32_t tag, rtag;            // words of exchange / reduction q carry tag + q (q from 1)
    unsigned long long* inbox;
    int stride;
    unsigned long long* rows;
    double* out;                   // its, stalled, BV_STATS values, exchanges, reductions
    unsigned int* err;
    unsigned polls;
};
constexpr int BV_CG_OUT = BV_STATS + 4;
constexpr int BV_RING = 2;
constexpr int BV_EVERY = 50;       // iterations between looks at the residual

__host__ __device__ constexpr int bv_cg_smem(int cpt) {
    return (cpt * RES_PLANE + 34) * (int)sizeof(double);
}

// One potential solve, -K phi = -bphi by conjugate gradients preconditioned with the diagonal,
// from the potential in `phi`; the iteration, its stopping rule and its checks are those of
// the launches (bv_cg_*): the true residual every 50 iterations, done at tol or at the
// rounding floor 64 eps max(diag |phi|), given up after 20 looks without a halving.
// Two reductions bound an iteration; the z values of the faces travel beside the second.
// T: most threads; up to 256 the compiler has 255 registers for a thread's state.
template <int CPT, int T>
__global__ void __launch_bounds__(T, 1) bv_cgr_kernel(const BVCgArgs A) {
    extern __shared__ double res_sd[];
    const int t = threadIdx.x;
    const BVArgs& B = A.B;
    ResBrick<CPT, BV_RING, 1> G;
    G.init(A.cut, A.stride);
    double* const S = res_sd;
    ResReduce R{A.rows, res_sd + CPT * RES_PLANE, A.rtag + 1, A.err, A.polls, true, false};
    auto plus = [](double a, double b) { return a + b; };
    const int64_t nxny = B.nxny;
    const int64_t c0 = G.i + (int64_t)B.nx * G.j + nxny * G.k0;
    const bool in_xy = G.mine && G.i < B.nx && G.j < B.ny;
    for (int q = t; q < CPT * RES_PLANE; q += (int)blockDim.x) S[q] = 0.0;

    // face conductivities kappa_f / h^2 (-x, +x, -y, +y; the column's z faces), the membrane's,
    // 1 / diagonal
    double kf[CPT][4], kz[CPT + 1], km[CPT], dinv[CPT], x[CPT], r[CPT], p[CPT];
    uint32_t fluid = 0;
#pragma unroll
    for (int e = 0; e < CPT; ++e) {
        const int64_t c = c0 + nxny * e;
        const unsigned f = in_xy && G.k0 + e < B.nz ? B.flags[c] : 0u;
        if (f & F_FLUID) fluid |= 1u << e;
        const bool fl = f & F_FLUID;
        const double kc = fl ? A.kcell[c] : 0.0;
        const unsigned bit[6] = {F_XM, F_XP, F_YM, F_YP, F_ZM, F_ZP};
        const int64_t off[6] = {-1, 1, -B.nx, B.nx, -nxny, nxny};
        double dg = 0.0;
#pragma unroll
        for (int m = 0; m < 6; ++m) {
            const double k = (f & bit[m]) ? 0.5 * (kc + A.kcell[c + off[m]]) / B.h2 : 0.0;
            if (m < 4) kf[e][m < 4 ? m : 0] = k;
            else if (m == 5) kz[e + 1] = k;
            else if (e == 0) kz[0] = k;                // the others: the face of the cell below
            dg += k;
        }
        km[e] = fl ? 2.0 * A.kmem[c] / B.h2 : 0.0;
        dg += km[e];
        dinv[e] = dg > 0.0 ? 1.0 / dg : 0.0;
        x[e] = fl ? A.phi[c] : 0.0;
    }
    uint32_t tag = A.tag;
    double zlo[1], zhi[1], ring[BV_RING];
    auto slot = [&]() { return A.inbox + 2 * ((tag & 1u) * A.stride); };
    // exchange: v of the faces to the neighbours, theirs into zlo, zhi and ring
    auto exchange_send = [&](const double (&v)[CPT]) {
        ++tag;
        G.send(slot(), v, tag);
    };
    auto exchange_poll = [&]() {
        zlo[0] = zhi[0] = 0.0;
        for (int m = 0; m < BV_RING; ++m) ring[m] = 0.0;
        __syncwarp();                  // the warp's own words are sent before it starts polling
        G.poll(slot(), A.stride, tag, zlo, zhi, ring, A.err, A.polls, R.good);
    };
    // A v for the column e, v in S with its neighbours
    auto apply = [&](int e, const double (&v)[CPT], double lo, double hi) {
        const double* P = S + e * RES_PLANE;
        const double vc = v[e];
        double a = kf[e][0] * (vc - P[G.oxm]);
        a = fma(kf[e][1], vc - P[G.oxp], a);
        a = fma(kf[e][2], vc - P[G.o - G.bx], a);
        a = fma(kf[e][3], vc - P[G.o + G.bx], a);
        a = fma(kz[e], vc - (e > 0 ? v[e > 0 ? e - 1 : 0] : lo), a);
        a = fma(kz[e + 1], vc - (e + 1 < CPT ? v[e + 1 < CPT ? e + 1 : e] : hi), a);
        return fma(km[e], vc, a);
    };
    // the true residual b - A x in res (x exchanged first), leaving S to the caller
    auto residual = [&](double (&res)[CPT]) {
        exchange_send(x);
        exchange_poll();
        __syncthreads();
        if (G.mine)
            for (int e = 0; e < CPT; ++e) S[e * RES_PLANE + G.o] = x[e];
#pragma unroll
        for (int m = 0; m < BV_RING; ++m)
            if (G.want & (4u << m)) S[G.dst[m]] = ring[m];
        __syncthreads();
#pragma unroll
        for (int e = 0; e < CPT; ++e)
            res[e] = (fluid >> e) & 1u
                         ? -A.bphi[c0 + nxny * e] - apply(e, x, zlo[0], zhi[0]) : 0.0;
        __syncthreads();
    };
    // the residual's largest entry, the largest change of phi, its sum, extremes, largest term
    double stats[BV_STATS];
    auto look = [&](const double (&res)[CPT]) {
        double s[BV_STATS] = {0.0, 0.0, 0.0, INFINITY, -INFINITY, 0.0};
#pragma unroll
        for (int e = 0; e < CPT; ++e) {
            if (!((fluid >> e) & 1u)) continue;
            s[0] = fmax(s[0], fabs(res[e]));
            s[1] = fmax(s[1], fabs(x[e] - A.phi[c0 + nxny * e]));   // phi: still the start's
            s[2] += x[e];
            s[3] = fmin(s[3], x[e]);
            s[4] = fmax(s[4], x[e]);
            s[5] = fmax(s[5], dinv[e] > 0.0 ? fabs(x[e]) / dinv[e] : 0.0);
        }
        // a NaN residual shows as an infinite one (fmax drops it)
#pragma unroll
        for (int e = 0; e < CPT; ++e)
            if (!isfinite(res[e])) s[0] = INFINITY;
#pragma unroll 1
        for (int q = 0; q < BV_STATS; ++q) {
            const double none = q == 3 ? INFINITY : q == 4 ? -INFINITY : 0.0;
            const double v = q == 0 ? s[0] : q == 1 ? s[1] : q == 2 ? s[2] : q == 3 ? s[3]
                                                                     : q == 4 ? s[4] : s[5];
            stats[q] = R.all(v, none, [q](double a, double b) {
                return q == 2 ? a + b : q == 3 ? fmin(a, b) : fmax(a, b);
            });
        }
    };
    auto done = [&]() { return stats[0] <= fmax(A.tol, 64.0 * 2.2e-16 * stats[5]); };

    double z[CPT];
    double plo = 0.0, phi_ = 0.0;                      // p below and above the column
    double pr[BV_RING];                                // p around the brick, kept over a look
#pragma unroll
    for (int m = 0; m < BV_RING; ++m) pr[m] = 0.0;
    // p from z (first: p = z) with beta, in the column, its halo and the shared ring
    auto direction = [&](double beta) {
#pragma unroll
        for (int e = 0; e < CPT; ++e) {
            p[e] = fma(beta, p[e], z[e]);
            if (G.mine) S[e * RES_PLANE + G.o] = p[e];
        }
        plo = fma(beta, plo, zlo[0]);
        phi_ = fma(beta, phi_, zhi[0]);
#pragma unroll
        for (int m = 0; m < BV_RING; ++m)
            if (G.want & (4u << m)) {
                pr[m] = fma(beta, pr[m], ring[m]);
                S[G.dst[m]] = pr[m];
            }
        __syncthreads();
    };
    int it = 0, stall = 0;
    double best = 0.0, rz = 0.0;
#pragma unroll
    for (int e = 0; e < CPT; ++e) p[e] = 0.0;
#pragma unroll 1
    for (bool first = true;; first = false) {
        residual(z);                                   // the true residual, in z for the moment
        look(z);
        if (!isfinite(stats[0])) break;
        if (first || stats[0] < 0.5 * best) {
            best = stats[0];
            stall = 0;
        } else {
            ++stall;
        }
        if (done() || it >= A.max_it || stall >= 20 || R.dead) break;
        // S holds phi: put p back, or (first) p = 0 and the start r = residual, p = z
        if (!first) {
#pragma unroll
            for (int e = 0; e < CPT; ++e)
                if (G.mine) S[e * RES_PLANE + G.o] = p[e];
#pragma unroll
            for (int m = 0; m < BV_RING; ++m)
                if (G.want & (4u << m)) S[G.dst[m]] = pr[m];
            __syncthreads();
        }
#pragma unroll 1
        for (int q = first ? -1 : 0; q < BV_EVERY && it < A.max_it && !R.dead; ++q) {
            double s = 0.0, alpha = 0.0, qv[CPT];
            if (q < 0) {
#pragma unroll
                for (int e = 0; e < CPT; ++e) {
                    r[e] = z[e];
                    qv[e] = 0.0;
                }
            } else {
                ++it;
#pragma unroll
                for (int e = 0; e < CPT; ++e) {
                    qv[e] = G.mine ? apply(e, p, plo, phi_) : 0.0;
                    s = fma(p[e], qv[e], s);
                }
                alpha = R.all(s, 0.0, plus, [&](double pq) { return pq != 0.0 ? rz / pq : 0.0; }).y;
            }
            s = 0.0;
#pragma unroll
            for (int e = 0; e < CPT; ++e) {
                x[e] = fma(alpha, p[e], x[e]);
                r[e] = fma(-alpha, qv[e], r[e]);
                z[e] = dinv[e] * r[e];
                s = fma(r[e], z[e], s);
            }
            exchange_send(z);
            const double2 zz =
                R.all(s, 0.0, plus, [&](double v) { return rz != 0.0 ? v / rz : 0.0; });
            exchange_poll();
            rz = zz.x;
            direction(zz.y);                           // first: rz and beta are 0
        }
    }
    // every CTA has read the start's phi: the reductions of the last look came after
#pragma unroll
    for (int e = 0; e < CPT; ++e)
        if ((fluid >> e) & 1u) A.phi[c0 + nxny * e] = x[e];
    if (blockIdx.x == 0 && t == 0) {
        A.out[0] = it;
        A.out[1] = stall;
        for (int q = 0; q < BV_STATS; ++q) A.out[2 + q] = stats[q];
        A.out[2 + BV_STATS] = tag - A.tag;             // exchanges and reductions made
        A.out[3 + BV_STATS] = R.tag - 1 - A.rtag;
    }
}

// ---------------------------------------------------------------------------------
// Species sweeps at a fixed potential. With phi fixed the right-hand side of a species at a
// cell is linear, d C_c + sum_f a_f C_f + b (+ n_j S), the source S = kf C_O - kb C_R and the
// steps are constant: they are formed once per launch from the expressions of bv_species_rhs
// and bv_source. The quinones have one diffusivity and charge, so they share a_f and d. About
// 30 FP64 operations a cell and sweep instead of some 270 (two exponentials, three divisions,
// the migration terms).
// ---------------------------------------------------------------------------------
struct BVSweepArgs {
    BVArgs B;
    ResCut cut;
    const double* __restrict__ phi;
    const double* C[3];            // O, R, H before the first sweep
    double* C2[3];                 // after the last (other buffers)
    int n;
    uint32_t tag;
    unsigned long long* inbox;
    int stride;
    unsigned int* err;
    unsigned polls;
};
constexpr int BVS_CPT = 2;         // cells of a column: 22 doubles each
__host__ __device__ constexpr int bv_sweep_smem() {
    return (2 * 3 * BVS_CPT * RES_PLANE + 7 * BVS_CPT * RES_T) * (int)sizeof(double);
}

template <int T>
__global__ void __launch_bounds__(T, 1) bv_sweepr_kernel(const BVSweepArgs A) {
    constexpr int CPT = BVS_CPT, copy = 3 * CPT * RES_PLANE;
    extern __shared__ double res_sd[];
    const int t = threadIdx.x;
    const BVArgs& B = A.B;
    ResBrick<CPT, BV_RING, 3> G;
    G.init(A.cut, A.stride);
    double* const hs = res_sd + 2 * copy + t;          // the protons' a_f and d
    const int64_t nxny = B.nxny;
    const int64_t c0 = G.i + (int64_t)B.nx * G.j + nxny * G.k0;
    const bool in_xy = G.mine && G.i < B.nx && G.j < B.ny;
    double aq[CPT][6], dq[CPT], step[CPT][3], kf[CPT], kb[CPT], C[CPT][3], bin[3] = {0, 0, 0};
    uint32_t fluid = 0;
#pragma unroll
    for (int e = 0; e < CPT; ++e) {
        const int64_t c = c0 + nxny * e;
        const unsigned f = in_xy && G.k0 + e < B.nz ? B.flags[c] : 0u;
        double dh = 0.0, ah[6];
        dq[e] = kf[e] = kb[e] = 0.0;
#pragma unroll
        for (int m = 0; m < 6; ++m) aq[e][m] = ah[m] = 0.0;
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            step[e][v] = 0.0;
            C[e][v] = in_xy && G.k0 + e < B.nz ? A.C[v][c] : 0.0;
        }
        if (f & F_FLUID) {
            fluid |= 1u << e;
            const BVCell b = bv_cell(B, c, f);
            const double pc = A.phi[c];
            bv_source(B, b, c, 0.0, 0.0, pc, &kf[e], &kb[e]);
            const BVSpecies &Q = B.sp[0], &P = B.sp[2];
            double out = 0.0, mdiag = 0.0;
#pragma unroll
            for (int m = 0; m < 6; ++m) {
                const double q = b.q[m];
                if (q > 0.0) out += q;
                if (b.n[m] >= 0) {
                    const double hd = 0.5 * (A.phi[b.n[m]] - pc), in = q > 0.0 ? 0.0 : -q;
                    aq[e][m] = in + Q.Dh + Q.g * hd;
                    ah[m] = in + P.Dh + P.g * hd;
                    mdiag += hd;
                }
            }
            const double mh = b.membrane ? mdiag - 2.0 * pc : mdiag;
            dq[e] = -out - Q.Dh * b.nf + Q.g * mdiag;
            dh = -out - P.Dh * b.nf + P.g * mh;
            double sq = out + Q.Dh * b.nf, sh = out + P.Dh * b.nf;
            if (b.inlet) {
                const double in = b.q[4] > 0.0 ? 0.0 : -b.q[4];
                dq[e] -= Q.gDh;
                dh -= P.gDh;
                sq += Q.gDh;
                sh += P.gDh;
#pragma unroll
                for (int v = 0; v < 3; ++v) bin[v] = (in + B.sp[v].gDh) * B.sp[v].c_in;
            }
            sq += fabs(Q.g * mdiag);
            sh += fabs(P.g * mh);
            step[e][0] = B.cfl / (sq + kf[e]);
            step[e][1] = B.cfl / (sq + kb[e]);
            step[e][2] = B.cfl / sh;
        }
#pragma unroll
        for (int m = 0; m < 6; ++m) hs[(7 * e + m) * RES_T] = ah[m];
        hs[(7 * e + 6) * RES_T] = dh;
    }
    // the brick and the columns around it before the first sweep (0 outside the lattice)
    for (int q = t; q < 2 * copy; q += (int)blockDim.x) {
        const int v = q % copy / (CPT * RES_PLANE), e = q % (CPT * RES_PLANE) / RES_PLANE;
        const int p = q % RES_PLANE, r = p % RES_ROWS;
        const int bx = A.cut.bx, by = A.cut.by, b = blockIdx.x;
        int yy = r / bx, xx = r % bx;
        bool at = q < copy;
        if (p >= RES_ROWS) {
            if (xx == bx - 1) { ++yy; xx = -1; }
            else if (xx == 0) { --yy; xx = bx; }
            else at = false;
            if (yy < 1 || yy > by) at = false;
        }
        const int gi = b % A.cut.gx * bx + xx, gj = (b / A.cut.gx) % A.cut.gy * by + yy - 1;
        const int gk = G.k0 + e;
        at = at && yy < by + 2 && gi >= 0 && gi < B.nx && gj >= 0 && gj < B.ny && gk < B.nz;
        res_sd[q] = at ? A.C[v][gi + (int64_t)B.nx * gj + nxny * gk] : 0.0;
    }
    double zlo[3], zhi[3], ring[BV_RING];
#pragma unroll
    for (int v = 0; v < 3; ++v) {
        zlo[v] = in_xy && G.k0 > 0 ? A.C[v][c0 - nxny] : 0.0;
        zhi[v] = in_xy && G.k0 + CPT < B.nz ? A.C[v][c0 + nxny * CPT] : 0.0;
    }
    bool good = true;
    __syncthreads();
    for (int ver = 1; ver <= A.n; ++ver) {
        const double* Sr = res_sd + ((ver - 1) & 1) * copy;
        double* Sw = res_sd + (ver & 1) * copy;
        const uint32_t tag = A.tag + (uint32_t)ver;
        unsigned long long* const slot = A.inbox + 2 * ((ver & 1) * 3 * A.stride);
        const bool more = ver < A.n;
        if (G.mine) {
            double N[3][CPT];
#pragma unroll
            for (int e = 0; e < CPT; ++e) {
                const double src = kf[e] * C[e][0] - kb[e] * C[e][1];
#pragma unroll
                for (int v = 0; v < 3; ++v) {
                    const double* P = Sr + (v * CPT + e) * RES_PLANE;
                    auto a = [&](int m) { return v < 2 ? aq[e][m] : hs[(7 * e + m) * RES_T]; };
                    const double zm = e > 0 ? C[e > 0 ? e - 1 : 0][v] : zlo[v];
                    const double zp = e + 1 < CPT ? C[e + 1 < CPT ? e + 1 : e][v] : zhi[v];
                    double r = (v < 2 ? dq[e] : hs[(7 * e + 6) * RES_T]) * C[e][v];
                    if (e == 0) r += bin[v];           // only the inlet plane's: k0 = 0
                    r = fma(a(0), P[G.oxm], r);
                    r = fma(a(1), P[G.oxp], r);
                    r = fma(a(2), P[G.o - G.bx], r);
                    r = fma(a(3), P[G.o + G.bx], r);
                    r = fma(a(4), zm, r);
                    r = fma(a(5), zp, r);
                    r = fma(B.sp[v].nst, src, r);
                    N[v][e] = fma(step[e][v], r, C[e][v]);
                }
            }
#pragma unroll
            for (int v = 0; v < 3; ++v) {
                if (more) G.send(slot + 2 * v * A.stride, N[v], tag);
#pragma unroll
                for (int e = 0; e < CPT; ++e) {
                    C[e][v] = N[v][e];
                    Sw[(v * CPT + e) * RES_PLANE + G.o] = N[v][e];
                }
            }
        }
        if (!more) break;
        __syncwarp();                  // the warp's own words are sent before it starts polling
        G.poll(slot, A.stride, tag, zlo, zhi, ring, A.err, A.polls, good);
#pragma unroll
        for (int m = 0; m < BV_RING; ++m)
            if (G.want & (4u << m)) Sw[G.dst[m]] = ring[m];
        __syncthreads();
    }
#pragma unroll
    for (int e = 0; e < CPT; ++e)
        if ((fluid >> e) & 1u)
#pragma unroll
            for (int v = 0; v < 3; ++v) A.C2[v][c0 + nxny * e] = C[e][v];
}

}  // namespace rfb
