// The Hartree CG with the separable preconditioner as one persistent cooperative kernel.
//
// As kernels of their own (ten launches with the six-pass preconditioner) an iteration's phases cost
// 112 us at 49^3 nodes, most of it launch latency, reloading the axis matrices and draining; here
// one CTA per SM keeps the six axis matrices, the stencil tables and its tensor memory for the whole
// solve, the phases are separated by grid barriers, and the residual test runs on the device after
// every iteration, so a solve is one launch and one host synchronization, and what it gives depends on
// U, the right-hand side and the tolerance alone.
//
// The iteration is Chronopoulos and Gear's arrangement of CG (J. Comput. Appl. Math. 25, 1989): the
// operator is applied to z = A_sep^-1 r instead of p, w = L z, and s = L p follows by recurrence,
//   beta = (r.z)' / (r.z),  alpha = r.z / (z.w - beta r.z / alpha_previous),
//   p = z + beta p,  s = w + beta s,  U += alpha p,  r -= alpha s,
// so both sums are known after one phase, and the four phases of an iteration are
//   middle pass | backward pass, r.z | SpMV, z.w | update and forward pass, r.r.
// p and U need only their own node, so CTAs without a plane of the forward pass take them (or, where
// few are left over, all CTAs behind their middle tiles).  z has float32 values, which halves the
// float-float SpMV's gathers.  A test that passes ends the solve before the middle pass.
//
// Measured against the usual arrangement (SpMV on p, five barriers), Hartree solves of four steps: 8^3
// cells 2.46 -> 2.38 ms, 24^3 3.41 -> 3.15, 21x19x23 3.40 -> 3.20, 60x32x30 (float-float) 4.45 -> 4.01.
// float64 operations of a warp take 16 cycles each, so the
// passes that run on few SMs hold as few of them as possible.  An iteration of a cold solve at 8^3, 24^3 and
// 60x32x30 cells takes 28.6, 39.5 and 77.9 us with 512 threads, 29.3, 44.8 and 106 with 256, 32.6, 44.4 and
// 84.6 with 768 (separate kernels: 72, 88 and 131).
//
// Sums over the grid go through one partial per CTA, written before a barrier and added in CTA
// order by every CTA after it.  A barrier wait is bounded: on timeout the CTA raises the abort
// flag, which every other wait polls, and the host returns OFKS_ETIMEOUT.
#include <algorithm>
#include <cmath>

#include "sep_plane.cuh"

namespace {

using namespace sepp;

constexpr int NTH = 512, NW = NTH / 32;
constexpr int BATCH = 8;                          // stencil entries whose loads are issued together
constexpr int SPLIT_ROW = 40;                     // rows of more entries are shared by two lanes
constexpr long long BAR_WAIT = 1LL << 21;
// At least half of an SM's shared memory, so that two solves on streams of their own never share an
// SM.  There, one solve's CTA could wait for tensor memory that the other's holds on one SM and hold
// what the other's waits for on another, both behind their grid barriers.  Other kernels that use
// tensor memory do not wait for other CTAs, so theirs is given back.
constexpr uint32_t ALONE = 114 * 1024;
constexpr int OWN = 20 * 1024;                    // at least the kernel's static shared memory

struct CgOut {
    double rr, bb;
    int it, status, abort;
    unsigned bar;
    unsigned long long ns[2];                     // profiling: nanoseconds of the SpMV, of the passes
};
static_assert(sizeof(CgOut) <= 8 * sizeof(double), "room in cg_loop_doubles");

struct Loop {
    int nx, ny, nz, px, py, pz, ncol, NT;
    const bf *S[3], *St[3];
    const float *lx, *lyzp;
    float *T;
    uint32_t oSt[3], oS[3], oB, part_p, part_m;   // shared-memory offsets; bytes per data part
    int tcols;
    Vecs V;
    double *p;
    float *zf;                                    // z, float32 (in the room of the float64 z; float-float SpMV)
    const double *rhs;
    double *q;                                    // w = L z
    int Lx;
    const StencilType *types;
    const StencilCode *code;
    const double *val;
    const float2 *valff;
    double tol2;
    int max_iter;
    int timed;                                    // profiling is on
    double *part;                                 // 4 x gridDim.x: zw, rr, rz, |rhs|^2
    CgOut *out;
};

// barrier over the grid; target counts this CTA's arrivals times the grid.  False after an abort.
__device__ __forceinline__ bool grid_barrier(CgOut *out, unsigned &target, int *s_abort) {
    __syncthreads();
    if (threadIdx.x == 0) {
        target += gridDim.x;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&out->bar) : "memory");
        bool ok = false;
        for (long long w = 0; w < BAR_WAIT; ++w) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&out->bar) : "memory");
            if ((int)(v - target) >= 0) { ok = true; break; }
            if ((w & 63) == 63 && *(volatile int *)&out->abort) break;
        }
        if (!ok) { atomicExch(&out->abort, 1); *s_abort = 1; }
    }
    __syncthreads();
    return *s_abort == 0;
}

// sum of the CTAs' partials in CTA order, by one warp of every CTA; the loads of the first 192 together
__device__ __forceinline__ double warp_total(const double *part) {
    constexpr int U = 6;
    const unsigned lane = threadIdx.x & 31;
    double v[U], s = 0.0;
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = lane + 32 * u < gridDim.x ? __ldcg(part + lane + 32 * u) : 0.0;
#pragma unroll
    for (int u = 0; u < U; ++u) s += v[u];
    for (unsigned i = lane + 32 * U; i < gridDim.x; i += 32) s += __ldcg(part + i);
    return warp_sum(s);
}

__device__ __forceinline__ double grid_total(const double *part, double *s_val) {
    if (threadIdx.x < 32) {
        const double s = warp_total(part);
        if (threadIdx.x == 0) *s_val = s;
    }
    __syncthreads();
    return *s_val;
}

// two such sums, one by each of the first two warps
__device__ __forceinline__ void grid_totals(const double *p0, const double *p1, double *s_two) {
    if (threadIdx.x < 64) {
        const double s = warp_total(threadIdx.x < 32 ? p0 : p1);
        if ((threadIdx.x & 31) == 0) s_two[threadIdx.x >> 5] = s;
    }
    __syncthreads();
}

struct Tables {
    StencilType type[8];
    StencilCode code[8 * ST_MAXE];
    int wblk[9];                                  // first block of each type (one warp's rows)
};

// a row of the stencil, or this lane's part of it: entries [e0, e1) of its type, its lattice
// position and node, and its index in the four parity classes
struct Row {
    int t, e0, e1, a, b, c, node, idx[4];
};

// the row's product with x over its entries in the order of the stencil kernels, BATCH loads at a time
template <class F2, class X2, class Get, class Acc>
__device__ __forceinline__ void row_product(const Tables &tb, const Row &R, const F2 *__restrict__ val, X2, Get get, Acc acc) {
    const StencilCode *se = tb.code + R.t * ST_MAXE;
    auto fetch = [&](const StencilCode &E, F2 &v, X2 &x) {
        const int lo = E.lin4 & 1 ? R.idx[1] : R.idx[0], hi = E.lin4 & 1 ? R.idx[3] : R.idx[2];
        v = __ldg(val + E.off + (E.lin4 & 2 ? hi : lo));
        x = get(R.node + (E.lin4 >> 2));
    };
    F2 v[BATCH];
    X2 x[BATCH];
    int e = R.e0;
    for (; e + BATCH <= R.e1; e += BATCH) {
#pragma unroll
        for (int u = 0; u < BATCH; ++u) fetch(se[e + u], v[u], x[u]);
#pragma unroll
        for (int u = 0; u < BATCH; ++u) acc(v[u], x[u]);
    }
#pragma unroll
    for (int u = 0; u < BATCH - 1; ++u)           // the rest, its loads together too
        if (e + u < R.e1) fetch(se[e + u], v[u], x[u]);
#pragma unroll
    for (int u = 0; u < BATCH - 1; ++u)
        if (e + u < R.e1) acc(v[u], x[u]);
}

__device__ __forceinline__ void ff_madd(float &sh, float &sl, const float2 a, const float x) {
    const float p = __fmul_rn(a.x, x);
    float e = __fmaf_rn(a.x, x, -p);
    e = __fmaf_rn(a.y, x, e);
    const float t = __fadd_rn(sh, p);
    const float bv = __fsub_rn(t, sh);
    const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bv)), __fsub_rn(p, bv));
    sh = t;
    sl = __fadd_rn(sl, __fadd_rn(err, e));
}

// Rows in blocks of one node type, 32 per warp or, where a row is long (cell vertices, 65 entries),
// 16 with two lanes to a row, dealt to the grid's CTAs in turn and within a CTA to the warps forth and
// back: s = product(row) over the row's interior entries, then done(row, s) on one lane per row
// (interior or not).
template <class Product, class Done>
__device__ __forceinline__ void for_rows(const Loop &P, const Tables &tb, Product product, Done done) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int round = 0; round * NW * (int)gridDim.x < tb.wblk[8]; ++round) {
        const int k = round * NW + (round & 1 ? NW - 1 - warp : warp);
        const int wb = k * (int)gridDim.x + (int)blockIdx.x;
        if (wb >= tb.wblk[8]) continue;           // the same for the whole warp
        int t = 0;
        while (wb >= tb.wblk[t + 1]) ++t;
        const StencilType &T = tb.type[t];
        const bool two = T.nent > SPLIT_ROW;
        const int idx = two ? (wb - tb.wblk[t]) * 16 + (lane & 15) : (wb - tb.wblk[t]) * 32 + lane;
        const int nyz = T.ny * T.nz, ia = idx / nyz, rem = idx - ia * nyz, ib = rem / T.nz, ic = rem - ib * T.nz;
        Row R;
        R.t = t; R.a = 2 * ia + T.px; R.b = 2 * ib + T.py; R.c = 2 * ic + T.pz;
        R.node = (R.a * P.V.Ly + R.b) * P.V.Lz + R.c;
        const int half = (T.nent + 1) >> 1;
        R.e0 = two && lane >= 16 ? half : 0;
        R.e1 = two && lane < 16 ? half : T.nent;
#pragma unroll
        for (int q = 0; q < 4; ++q) {             // class q: extents of the sub-lattices of that parity
            const int ny = (P.V.Ly - (q >> 1) + 1) >> 1, nz = (P.V.Lz - (q & 1) + 1) >> 1;
            R.idx[q] = (ia * ny + ib) * nz + ic;
        }
        const bool in = idx < T.n && R.a > 0 && R.a < P.Lx - 1 && R.b > 0 && R.b < P.V.Ly - 1 && R.c > 0 && R.c < P.V.Lz - 1;
        double s = in ? product(R) : 0.0;
        if (two) s += __shfl_xor_sync(0xffffffffu, s, 16);
        if (idx < T.n && (!two || lane < 16)) done(R, in, s);
    }
}

template <int FF>
__global__ void __launch_bounds__(NTH, 1) k_cg_loop(const Loop P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ Tables tb;
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag, s_abort;
    __shared__ double sh[NW], s_val, s_two[2], s_ab[2];
    __shared__ float s_l[64];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned G = gridDim.x;
    const uint32_t sm = su32(dsm), sB = sm + P.oB;
    const int mtx = (P.px + 127) >> 7, mty = (P.py + 127) >> 7, mtz = (P.pz + 127) >> 7;
    double *part_zw = P.part, *part_rr = P.part + G, *part_rz = P.part + 2 * G, *part_bb = P.part + 3 * G;
    for (int i = threadIdx.x; i < 8 * ST_MAXE; i += NTH) tb.code[i] = P.code[i];
    if (threadIdx.x < 8) tb.type[threadIdx.x] = P.types[threadIdx.x];
    if (threadIdx.x == 0) {
        int w = 0;
        for (int t = 0; t < 8; ++t) { tb.wblk[t] = w; const int per = P.types[t].nent > SPLIT_ROW ? 16 : 32; w += ((int)P.types[t].n + per - 1) / per; }
        tb.wblk[8] = w;
        s_abort = 0;
    }
    load_axis<NW>(sm + P.oSt[0], P.St[0], P.px); load_axis<NW>(sm + P.oS[0], P.S[0], P.px);
    load_axis<NW>(sm + P.oSt[1], P.St[1], P.py); load_axis<NW>(sm + P.oS[1], P.S[1], P.py);
    load_axis<NW>(sm + P.oSt[2], P.St[2], P.pz); load_axis<NW>(sm + P.oS[2], P.S[2], P.pz);
    Cta c;
    cta_open(c, &mbar, &tmem_base, &abort_flag, P.tcols);
    unsigned target = 0;
    bool ok = true;

    // r = rhs - L U, zero on the boundary, where z and p stay zero too
    {
        double rr = 0.0, bb = 0.0;
        for_rows(P, tb,
                 [&](const Row &R) {
                     double s = 0.0;
                     row_product(tb, R, P.val, 0.0, [&](int j) { return P.V.U[j]; }, [&](double v, double x) { s = fma(v, x, s); });
                     return s;
                 },
                 [&](const Row &R, bool in, double s) {
                     if (!in) {
                         P.V.r[R.node] = 0.0; P.p[R.node] = 0.0;
                         if (FF) P.zf[R.node] = 0.f; else P.V.z[R.node] = 0.0;
                         return;
                     }
                     const double f = P.rhs[R.node], ri = f - s;
                     P.V.r[R.node] = ri;
                     rr = fma(ri, ri, rr);
                     bb = fma(f, f, bb);
                 });
        const double t0 = cta_sum<NW>(rr, sh);
        __syncthreads();
        const double t1 = cta_sum<NW>(bb, sh);
        if (threadIdx.x == 0) { part_rr[blockIdx.x] = t0; part_bb[blockIdx.x] = t1; }
    }
    ok = grid_barrier(P.out, target, &s_abort);
    const double bb = grid_total(part_bb, &s_val);
    __syncthreads();
    double rr = grid_total(part_rr, &s_val), rz = 0.0;
    int it = 0, status = OFKS_OK;

    // p = z + beta p, U += alpha p on the interior (warps over the rows along c) by CTAs c0, c0 + 1, ...
    auto direction = [&](double alpha, double beta, int c0) {
        const int nc = (int)G - c0;
        if ((int)blockIdx.x < c0) return;
        for (int row = warp * nc + (int)blockIdx.x - c0; row < P.nx * P.ny; row += NW * nc) {
            const int a = row / P.ny, b = row - a * P.ny;
            const int o = ((a + 1) * P.V.Ly + (b + 1)) * P.V.Lz + 1;
            for (int cc = lane; cc < P.nz; cc += 32) {
                double v = FF ? f2d_bits(P.zf[o + cc]) : P.V.z[o + cc];
                if (beta != 0.0) v = fma(beta, P.p[o + cc], v);
                P.p[o + cc] = v;
                P.V.U[o + cc] = fma(alpha, v, P.V.U[o + cc]);
            }
        }
    };
    // forward pass; with update the CG update of s and r first, leaving r.r's partials (and p and U, where
    // at least half of the CTAs have no plane)
    const bool spare = (int)G >= 2 * P.nx;
    auto forward = [&](bool update, double alpha, double beta) -> bool {
        double prr = 0.0;
        bool good = true;
        for (int a = blockIdx.x; a < P.nx && good; a += G) {
            if (update) residual_to_data<NW, 2>(P.V, a, P.ny, P.nz, P.py, P.pz, alpha, beta, prr, dsm, P.oB, P.part_p);
            else residual_to_data<NW, 0>(P.V, a, P.ny, P.nz, P.py, P.pz, 0.0, 0.0, prr, dsm, P.oB, P.part_p);
            good = contract(c, sm + P.oSt[2], sB, P.part_p, mtz, P.py, P.pz);
            if (!good) break;
            acc_to_data<NW>(c, mtz, P.py, P.pz, sB, P.part_p);
            good = contract(c, sm + P.oSt[1], sB, P.part_p, mty, P.pz, P.py);
            if (!good) break;
            acc_to_global<NW>(c, mty, P.pz, P.ny, P.pz, P.T + (int64_t)a * P.ny * P.pz, P.pz);
        }
        if (update) {
            if (spare) direction(alpha, beta, P.nx);
            const double t = cta_sum<NW>(prr, sh);
            if (threadIdx.x == 0) part_rr[blockIdx.x] = t;
        }
        if (!good && threadIdx.x == 0) { s_abort = 1; atomicExch(&P.out->abort, 1); }
        return grid_barrier(P.out, target, &s_abort);
    };
    // middle and backward pass: z, r.z's partials.  With pending the last update's p and U come between them.
    auto backward = [&](bool pending, double alpha, double beta) -> bool {
        double prz = 0.0;
        bool good = true;
        for (int m0 = (int)blockIdx.x * P.NT; m0 < P.ncol && good; m0 += (int)G * P.NT) {
            mid_scales(P.lyzp, m0, P.ncol, P.NT, s_l);
            global_to_data<NW>(P.T + m0, P.ncol, P.nx, P.ncol - m0, P.NT, P.px, sB, P.part_m);
            good = contract(c, sm + P.oSt[0], sB, P.part_m, mtx, P.NT, P.px);
            if (!good) break;
            mid_scale<NW>(c, mtx, P.NT, P.nx, P.px, P.lx, s_l, dsm, P.oB, P.part_m);
            good = contract(c, sm + P.oS[0], sB, P.part_m, mtx, P.NT, P.px);
            if (!good) break;
            acc_to_global<NW>(c, mtx, P.NT, P.nx, P.ncol - m0, P.T + m0, P.ncol);
        }
        if (pending) direction(alpha, beta, 0);
        if (!good && threadIdx.x == 0) { s_abort = 1; atomicExch(&P.out->abort, 1); }
        if (!grid_barrier(P.out, target, &s_abort)) return false;
        for (int a = blockIdx.x; a < P.nx && good; a += G) {
            global_to_data<NW>(P.T + (int64_t)a * P.ny * P.pz, P.pz, P.ny, P.pz, P.pz, P.py, sB, P.part_p);
            good = contract(c, sm + P.oS[1], sB, P.part_p, mty, P.pz, P.py);
            if (!good) break;
            acc_to_data<NW>(c, mty, P.pz, P.py, sB, P.part_p);
            good = contract(c, sm + P.oS[2], sB, P.part_p, mtz, P.py, P.pz);
            if (!good) break;
            acc_to_z<NW, FF>(c, mtz, P.V, a, P.ny, P.nz, P.py, P.zf, nullptr, nullptr, prz);
        }
        const double t = cta_sum<NW>(prz, sh);
        if (threadIdx.x == 0) part_rz[blockIdx.x] = t;
        if (!good && threadIdx.x == 0) { s_abort = 1; atomicExch(&P.out->abort, 1); }
        return grid_barrier(P.out, target, &s_abort);
    };

    // profiling: the time since the last call goes to phase k, by one thread of the grid
    unsigned long long t_last = 0, t_ns[2] = {0, 0};
    const bool clock = P.timed && blockIdx.x == 0 && threadIdx.x == 0;
    auto lap = [&](int k) {
        if (!clock) return;
        unsigned long long t;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        if (k >= 0) t_ns[k] += t - t_last;
        t_last = t;
    };

    double alpha = 0.0, beta = 0.0;
    bool pending = false;
    lap(-1);
    while (ok) {
        // the residual test, before every iteration: its sum is complete behind the last barrier
        if (!isfinite(rr)) { status = OFKS_ENONFINITE; break; }
        if (rr <= P.tol2 * bb || bb == 0.0) break;
        if (it >= P.max_iter) { status = OFKS_ETIMEOUT; break; }
        if (it == 0 && !(ok = forward(false, 0.0, 0.0))) break;
        if (!(ok = backward(pending, alpha, beta))) break;
        pending = false;
        lap(1);
        double zw = 0.0;
        for_rows(P, tb,
                 [&](const Row &R) {
                     if constexpr (FF) {
                         float s_hi = 0.f, s_lo = 0.f;
                         row_product(tb, R, P.valff, 0.f, [&](int i) { return P.zf[i]; },
                                     [&](float2 v, float x) { ff_madd(s_hi, s_lo, v, x); });
                         return (double)s_hi + (double)s_lo;
                     } else {
                         double s = 0.0;
                         row_product(tb, R, P.val, 0.0, [&](int i) { return P.V.z[i]; },
                                     [&](double v, double x) { s = fma(v, x, s); });
                         return s;
                     }
                 },
                 [&](const Row &R, bool in, double s) {
                     if (!in) return;
                     P.q[R.node] = s;
                     zw = fma(FF ? f2d_bits(P.zf[R.node]) : P.V.z[R.node], s, zw);
                 });
        const double tzw = cta_sum<NW>(zw, sh);
        if (threadIdx.x == 0) part_zw[blockIdx.x] = tzw;
        if (!(ok = grid_barrier(P.out, target, &s_abort))) break;
        lap(0);
        grid_totals(part_rz, part_zw, s_two);
        if (threadIdx.x == 0) {
            double b = it > 0 ? s_two[0] / rz : 0.0;
            double den = it > 0 ? s_two[1] - b * s_two[0] / alpha : s_two[1];
            if (!(den > 0.0)) { b = 0.0; den = s_two[1]; }   // the recurrence is lost: again from p = z
            s_ab[0] = s_two[0] > 0.0 && den > 0.0 ? s_two[0] / den : 0.0;
            s_ab[1] = b;
        }
        __syncthreads();
        rz = s_two[0];
        alpha = s_ab[0];
        beta = s_ab[1];
        // no descent along z either (r.z or z.w not positive: z has no value beside its rounding, or r is
        // beyond float32): nothing that follows would differ
        if (alpha == 0.0) { status = isfinite(s_two[0]) && isfinite(s_two[1]) ? OFKS_ETIMEOUT : OFKS_ENONFINITE; break; }
        ok = forward(true, alpha, beta);
        pending = !spare;
        ++it;
        if (ok) rr = grid_total(part_rr, &s_val);
        __syncthreads();
        lap(1);
    }
    if (ok && pending) direction(alpha, beta, 0);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        P.out->rr = rr; P.out->bb = bb; P.out->it = it; P.out->status = status;
        P.out->ns[0] = t_ns[0]; P.out->ns[1] = t_ns[1];
    }
    cta_close(c, P.tcols, &P.out->abort);
}

// shared memory of the loop kernel; 0 when the operands do not fit
int place_loop(const SepState &S, Loop &P) {
    P.nx = S.n[0]; P.ny = S.n[1]; P.nz = S.n[2];
    P.px = pad16(P.nx); P.py = pad16(P.ny); P.pz = pad16(P.nz);
    P.ncol = P.ny * P.pz;
    P.NT = (P.ncol + 31) / 32 >= 100 ? ((P.ncol + 63) / 64 >= 120 ? 64 : 32) : 16;
    const int pad[3] = {P.px, P.py, P.pz};
    uint32_t o = 0;
    for (int d = 0; d < 3; ++d) {
        P.S[d] = S.hS[d]; P.St[d] = S.hSt[d];
        P.oSt[d] = o; o += axis_bytes(pad[d]);
        P.oS[d] = o; o += axis_bytes(pad[d]);
    }
    P.oB = o;
    P.part_p = data_bytes(P.py, P.pz);
    P.part_m = data_bytes(P.NT, P.px);
    P.lx = S.lx; P.lyzp = S.lyzp; P.T = S.t0;
    P.tcols = cols_of(std::max({tiles128(P.px) * P.NT, tiles128(P.pz) * P.py, tiles128(P.py) * P.pz}));
    const uint32_t need = o + 2 * std::max(P.part_p, P.part_m);
    return need <= (uint32_t)(SMEM_MAX - OWN) && P.tcols <= 512 ? (int)std::max(need, ALONE) : 0;
}

}  // namespace

// room for the result record and the partials
int64_t cg_loop_doubles(int sms) { return 8 + 4 * (int64_t)sms; }

// the persistent form applies: its operands fit in an SM's shared memory (axes of about 100
// interior points) and the mesh is small enough for launches to matter
bool cg_loop_fits(const SepState &S) {
    Loop P{};
    return S.plane && (int64_t)S.n[0] * S.n[1] * S.n[2] <= CG_LOOP_MAX_N && place_loop(S, P) > 0;
}

// Solves L U = rhs on the interior from U's current values and boundary data to
// |r|^2 <= tol2 |rhs|^2; iterations and status (OFKS_OK, OFKS_ETIMEOUT at max_iter,
// OFKS_ENONFINITE, or an error) on return.  One launch, one synchronization.  *ran is false, and nothing is
// done, where the device does not take the grid at once (fewer SMs at hand than it reports).
int cg_loop_run(ofks_ctx *c, double tol2, bool *ran, int *iters, int *status, double *rel2) {
    SepState &S = c->sep;
    Loop P{};
    const int smem = place_loop(S, P);
    P.V = {c->st.Ly, c->st.Lz, c->d_cp, c->d_cq, c->d_U, c->d_cr, c->d_cz, reinterpret_cast<double *>(c->d_cpff)};
    P.p = c->d_cp; P.zf = reinterpret_cast<float *>(c->d_cz); P.q = c->d_cq; P.rhs = c->d_rhs;
    P.Lx = c->st.Lx;
    P.types = c->st.d_type; P.code = c->st.d_code; P.val = c->st.val; P.valff = c->st.valff;
    P.tol2 = tol2; P.max_iter = c->prm.poisson_max_iter; P.timed = c->prof ? 1 : 0;
    P.out = reinterpret_cast<CgOut *>(S.loop_buf);
    P.part = S.loop_buf + 8;
    // CTAs: one per SM, fewer where the mesh has too few planes, tiles and rows to feed them
    const int64_t rows = c->n_nodes;
    const int want = std::max({P.nx, (P.ncol + P.NT - 1) / P.NT, (int)std::min<int64_t>(1 << 20, (rows + NTH - 1) / NTH)});
    const int grid = std::min(S.sms, want);
    auto kern = c->hartree_ff ? k_cg_loop<1> : k_cg_loop<0>;
    cudaError_t e = ofks_allow_smem((const void *)kern, OWN);
    if (e == cudaSuccess) e = cudaMemsetAsync(S.loop_buf, 0, sizeof(double) * 8, c->stream);
    void *args[] = {&P};
    if (e == cudaSuccess) e = cudaLaunchCooperativeKernel(kern, dim3((unsigned)grid), dim3(NTH), args, smem, c->stream);
    *ran = e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorNotSupported;
    if (!*ran) {
        cudaGetLastError();
        return OFKS_OK;
    }
    c->kernels += 1;
    CgOut h;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, P.out, sizeof(h), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return ofks_cuda_check(c, e, "Hartree CG");
    if (h.abort) return ofks_fail(c, OFKS_ETIMEOUT, "Hartree CG: a bounded device wait timed out");
    if (c->prof) {                                // the phases of the one launch, by the device's clock
        c->prof_n[PF_POISSON_SPMV] += h.it; c->prof_ms[PF_POISSON_SPMV] += 1e-6 * (double)h.ns[0];
        c->prof_n[PF_POISSON_PC] += h.it; c->prof_ms[PF_POISSON_PC] += 1e-6 * (double)h.ns[1];
    }
    *iters = h.it;
    *status = h.status;
    *rel2 = h.bb > 0.0 ? h.rr / h.bb : 0.0;
    return OFKS_OK;
}
