// Device code of the separable operator's inverse in three passes (sep_plane.cu, cg_loop.cu).
//
// z = (Sx (x) Sy (x) Sz) diag(1 / (lam_x + lam_y + lam_z)) (Sx (x) Sy (x) Sz)^T r is six dense
// contractions.  The two along y and z need only one x-plane of the tensor at a time, and the two
// along x (with the scaling between them) only one set of (y, z) columns, so
//   forward   per x-plane: contraction along z, then along y
//   middle    per tile of (y, z) columns: along x, the scaling, back along x
//   backward  per x-plane: back along y, then along z
// and the tensor crosses memory twice between the passes instead of five times.
//
// Operands are bf16 in the no-swizzle K-major core-matrix layout, the accumulators float32 in
// tensor memory.  The tensor's high and low bf16 parts (~16 significant bits, two MMAs per K step)
// are the B operand, [column n][k] with the contracted index k innermost; the axis matrix is the A
// operand, 128 rows per MMA, one or two row tiles (axes up to 256).  An accumulator row is one
// output index of the contraction; in the passes over planes a thread's 16 columns of it are
// consecutive k of the next operand (16-byte shared stores), in the middle pass lanes are
// consecutive k, so neighbouring lanes exchange a value and store pairs.  Core matrices of the
// data operands are 144 bytes apart along K, which keeps these stores off one bank.  Between the
// passes the tensor is float32, [a][j][pz] with rows of pz (nz rounded up to 16, padding zero).
//
// Waits are bounded: on timeout the CTA flags an error, frees its tensor memory and returns.
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"
#include "internal.h"

namespace sepp {

constexpr long long WAIT = 1LL << 20;
constexpr int LBA = 128, LBD = 144;               // bytes between core matrices along K: axis, data
constexpr int SMEM_MAX = 227 * 1024;

typedef __nv_bfloat16 bf;

__device__ __forceinline__ uint32_t su32(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// byte offset of element (r, k) of an operand with kc8 core matrices along K, LB bytes apart
template <int LB>
__device__ __forceinline__ uint32_t coff(int r, int k, int kc8) {
    return (uint32_t)(((r >> 3) * kc8 + (k >> 3)) * LB + (r & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ void cp16(uint32_t dst, const void *src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}

__device__ __forceinline__ void st16(uint32_t dst, uint4 v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

__device__ __forceinline__ uint32_t pack2(bf a, bf b) {
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// eight float32 values as bf16 high parts and their rounding errors as low parts
__device__ __forceinline__ void split8(const float *v, uint4 &hi, uint4 &lo) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bf a = __float2bfloat16(v[2 * i]), b = __float2bfloat16(v[2 * i + 1]);
        h[i] = pack2(a, b);
        l[i] = pack2(__float2bfloat16(v[2 * i] - __bfloat162float(a)),
                     __float2bfloat16(v[2 * i + 1] - __bfloat162float(b)));
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

__device__ __forceinline__ void tmem_ld16(uint32_t addr, float *v) {
    uint32_t u[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15}, [%16];"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]), "=r"(u[8]),
          "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(u[i]);
}

// double -> float by the bits (to nearest, ties away from zero), and float -> double (subnormals are zero in both):
// GB300's float64 unit takes 16 cycles for a warp's conversion, as long as for its multiply-add, and
// the values only feed operands of 16 significant bits or come from float32 sums
__device__ __forceinline__ float d2f_bits(double d) {
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const uint32_t e = (hi >> 20) & 0x7ffu, sign = hi & 0x80000000u;
    uint32_t m = ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
    m += (lo >> 28) & 1u;
    if (e < 897u) m = 0u;
    if (e > 1150u) m = e == 0x7ffu && ((hi & 0xfffffu) | lo) ? 0x7fffffffu : 0x7f800000u;
    return __uint_as_float(sign | m);
}

__device__ __forceinline__ double f2d_bits(float f) {
    const uint32_t b = __float_as_uint(f), e = (b >> 23) & 0xffu;
    uint32_t hi = (e == 0xffu ? 0x7ff00000u : (e + 896u) << 20) | ((b >> 3) & 0xfffffu);
    uint32_t lo = b << 29;
    if (e == 0u) hi = lo = 0u;
    return __hiloint2double((int)((b & 0x80000000u) | hi), (int)lo);
}

// sum over the block by its first warp, valid in thread 0; `sh` holds a double per warp
template <int NW>
__device__ __forceinline__ double cta_sum(double v, double *sh) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x >= 32) return 0.0;
    return warp_sum(threadIdx.x < NW ? sh[threadIdx.x] : 0.0);
}

// shared state of a CTA: barrier, tensor-memory base, abort flag; phase counts the commits
struct Cta {
    uint32_t tmem, mbar;
    int *abort_flag;
    uint32_t phase;
};

// D[mt][128 rows][N] = A (axis matrix, mt row tiles) times B (high + low data parts)^T, K = 16 ksteps,
// issued by one thread; every thread waits for the commit.  False after a timeout (uniform).
__device__ __forceinline__ bool contract(Cta &c, uint32_t a, uint32_t b, uint32_t part, int mt, int N, int K) {
    const int kc8 = K >> 3;
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (threadIdx.x == 0) {
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | (8u << 24);
        for (int t = 0; t < mt; ++t)
            for (int p = 0; p < 2; ++p)
                for (int kk = 0; kk < (K >> 4); ++kk) {
                    const uint64_t ad = sdesc(a + (uint32_t)(t * 16 * kc8 * LBA + kk * 2 * LBA), LBA, kc8 * LBA);
                    const uint64_t bd = sdesc(b + p * part + (uint32_t)(kk * 2 * LBD), LBD, kc8 * LBD);
                    const uint32_t accum = (p > 0 || kk > 0) ? 1u : 0u;
                    asm volatile(
                        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(c.tmem + t * N),
                        "l"(ad), "l"(bd), "r"(idesc), "r"(accum));
                }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(c.mbar));
    }
    uint32_t done = 0;
    for (long long w = 0; w < WAIT && !done; ++w)
        asm volatile(
            "{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}\n"
            : "=r"(done)
            : "r"(c.mbar), "r"(c.phase & 1));
    c.phase++;
    if (!done) *c.abort_flag = 1;
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    return *c.abort_flag == 0;
}

// tensor memory and barrier of the CTA; ends with a barrier
__device__ __forceinline__ void cta_open(Cta &c, uint64_t *mbar, uint32_t *tmem_base, int *abort_flag, int tcols) {
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_base)),
                     "r"(tcols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(mbar)));
        asm volatile("fence.mbarrier_init.release.cluster;");
        *abort_flag = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    c.tmem = *tmem_base;
    c.mbar = su32(mbar);
    c.abort_flag = abort_flag;
    c.phase = 0;
}

// after a timeout the MMAs of the last commit may still run: one more bounded wait before the
// tensor memory is released
__device__ __forceinline__ void cta_close(Cta &c, int tcols, int *err) {
    if (*c.abort_flag && threadIdx.x == 0) {
        atomicExch(err, 1);
        uint32_t done = 0;
        for (long long w = 0; w < WAIT && !done; ++w)
            asm volatile(
                "{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}\n"
                : "=r"(done)
                : "r"(c.mbar), "r"((c.phase - 1) & 1));
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(c.tmem), "r"(tcols));
}

// axis matrix (P x P, row-major, P a multiple of 16) into its operand at dst.  Rows past P of the
// last 128-row tile are left as they are: they only reach accumulator rows that are not read.
template <int NW>
__device__ void load_axis(uint32_t dst, const bf *__restrict__ S, int P) {
    const int kc8 = P >> 3;
    for (int r = threadIdx.x >> 3; r < P; r += NW * 4)
        for (int q = threadIdx.x & 7; q < kc8; q += 8) cp16(dst + coff<LBA>(r, q * 8, kc8), S + (int64_t)r * P + q * 8, 16);
}

// accumulator (rows r < rows of mt tiles, N columns) -> data operand (n = r, k = column), both parts
template <int NW>
__device__ __forceinline__ void acc_to_data(const Cta &c, int mt, int N, int rows, uint32_t dst, uint32_t part) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nc = N >> 4, k8 = N >> 3;
    for (int e = warp >> 2; e < mt * nc; e += NW >> 2) {
        const int t = e / nc, cb = (e - t * nc) << 4;
        const int r = t * 128 + (warp & 3) * 32 + lane;
        float v[16];
        tmem_ld16(c.tmem + t * N + cb + ((uint32_t)((warp & 3) * 32) << 16), v);
        if (r < rows)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint4 hi, lo;
                split8(v + 8 * h, hi, lo);
                const uint32_t o = dst + coff<LBD>(r, cb + 8 * h, k8);
                st16(o, hi);
                st16(o + part, lo);
            }
    }
}

// accumulator (rows r < rows, N columns) -> T[r ld + column], float32
template <int NW>
__device__ __forceinline__ void acc_to_global(const Cta &c, int mt, int N, int rows, int cols, float *T, int64_t ld) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nc = N >> 4;
    for (int e = warp >> 2; e < mt * nc; e += NW >> 2) {
        const int t = e / nc, cb = (e - t * nc) << 4;
        const int r = t * 128 + (warp & 3) * 32 + lane;
        float v[16];
        tmem_ld16(c.tmem + t * N + cb + ((uint32_t)((warp & 3) * 32) << 16), v);
        if (r < rows && cb < cols) {                  // cols is a multiple of 16
            float4 *d = reinterpret_cast<float4 *>(T + (int64_t)r * ld + cb);
#pragma unroll
            for (int h = 0; h < 4; ++h) d[h] = make_float4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
        }
    }
}

// T[r ld + n] (r < rows, n < cols, zero beyond) -> data operand (n, k = r), K rows of it: lanes
// along n, eight r per thread
template <int NW>
__device__ __forceinline__ void global_to_data(const float *T, int64_t ld, int rows, int cols, int N, int K,
                                               uint32_t dst, uint32_t part) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k8 = K >> 3, nn = (N + 31) >> 5;
    for (int e = warp; e < k8 * nn; e += NW) {
        const int q = e / nn, n = ((e - q * nn) << 5) + lane;
        if (n >= N) continue;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = (8 * q + i < rows && n < cols) ? T[(int64_t)(8 * q + i) * ld + n] : 0.f;
        uint4 hi, lo;
        split8(v, hi, lo);
        const uint32_t o = dst + coff<LBD>(n, 8 * q, k8);
        st16(o, hi);
        st16(o + part, lo);
    }
}

// the CG vectors on the lattice (all nodes, id = (a Ly + b) Lz + c)
struct Vecs {
    int Ly, Lz;
    const double *p, *q;
    double *U, *r, *z;
    double *s;
};

// plane a of the residual -> data operand (n = b, k = c), zero outside the interior.  With UPDATE 1 the
// CG update r -= alpha q, U += alpha p, rr += r.r comes first, with UPDATE 2 that of the single-reduction
// form (cg_loop.cu), s = q + beta s, r -= alpha s, rr += r.r.
template <int NW, int UPDATE>
__device__ __forceinline__ void residual_to_data(const Vecs &V, int a, int ny, int nz, int py, int pz, double alpha, double beta,
                                                 double &rr, unsigned char *dsm, uint32_t off, uint32_t part) {
    constexpr int FULL = UPDATE == 1;
    constexpr int PIECES = UPDATE ? 4 : 6;         // pieces of 32 values whose loads are issued together
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k8 = pz >> 3, nch = (pz + 31) >> 5;
    for (int e0 = warp; e0 < py * nch; e0 += NW * PIECES) {
        double rv[PIECES], pv[PIECES], qv[PIECES], uv[PIECES], sv[PIECES];
        int bb[PIECES], cc[PIECES];
        int64_t at[PIECES];
        bool in[PIECES];
#pragma unroll
        for (int u = 0; u < PIECES; ++u) {
            const int e = e0 + u * NW;
            bb[u] = e / nch;
            cc[u] = ((e - bb[u] * nch) << 5) + lane;
            in[u] = bb[u] < ny && cc[u] < nz;
            at[u] = ((int64_t)(a + 1) * V.Ly + (bb[u] + 1)) * V.Lz + 1 + cc[u];
            rv[u] = in[u] ? V.r[at[u]] : 0.0;
            if (UPDATE) qv[u] = in[u] ? V.q[at[u]] : 0.0;
            if (UPDATE == 2) sv[u] = in[u] && beta != 0.0 ? V.s[at[u]] : 0.0;
            if (FULL) pv[u] = in[u] ? V.p[at[u]] : 0.0;
            if (FULL) uv[u] = in[u] ? V.U[at[u]] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < PIECES; ++u) {
            if (bb[u] >= py || cc[u] >= pz) continue;
            double ri = rv[u];
            if (UPDATE && in[u]) {
                if (FULL) V.U[at[u]] = fma(alpha, pv[u], uv[u]);
                if (UPDATE == 2) {
                    if (beta != 0.0) qv[u] = fma(beta, sv[u], qv[u]);
                    V.s[at[u]] = qv[u];
                }
                ri = fma(-alpha, qv[u], ri);
                V.r[at[u]] = ri;
                rr = fma(ri, ri, rr);
            }
            const float f = d2f_bits(ri);
            const bf hi = __float2bfloat16(f);
            const uint32_t o = off + coff<LBD>(bb[u], cc[u], k8);
            *reinterpret_cast<bf *>(dsm + o) = hi;
            *reinterpret_cast<bf *>(dsm + o + part) = __float2bfloat16(f - __bfloat162float(hi));
        }
    }
}

// accumulator row c, columns b -> z of plane a, rz += r.z.  ZF: z as float32 (zf), else float64 (V.z,
// with pw also p, with pf p's float32 pairs).
template <int NW, int ZF>
__device__ __forceinline__ void acc_to_z(const Cta &c, int mtz, const Vecs &V, int a, int ny, int nz, int py, float *zf,
                                         double *pw, float2 *pf, double &rz) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nc = py >> 4;
    for (int e = warp >> 2; e < mtz * nc; e += NW >> 2) {
        const int t = e / nc, cb = (e - t * nc) << 4;
        const int cc = t * 128 + (warp & 3) * 32 + lane;
        double rv[16];
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i)
            rv[i] = (cc < nz && cb + i < ny) ? V.r[((int64_t)(a + 1) * V.Ly + (cb + i + 1)) * V.Lz + cc + 1] : 0.0;
        tmem_ld16(c.tmem + t * py + cb + ((uint32_t)((warp & 3) * 32) << 16), v);
        if (cc < nz)
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                if (cb + i >= ny) continue;
                const int64_t o = ((int64_t)(a + 1) * V.Ly + (cb + i + 1)) * V.Lz + cc + 1;
                const double zi = f2d_bits(v[i]);
                if (ZF) zf[o] = v[i];
                else {
                    V.z[o] = zi;
                    if (pw) pw[o] = zi;
                    if (pf) pf[o] = make_float2(v[i], 0.f);
                }
                rz = fma(rv[i], zi, rz);
            }
    }
}

// eigenvalues lam_y + lam_z of the tile's NT columns (1e30 past the end) into s_l
__device__ __forceinline__ void mid_scales(const float *lyzp, int m0, int ncol, int NT, float *s_l) {
    if ((int)threadIdx.x < NT) s_l[threadIdx.x] = m0 + (int)threadIdx.x < ncol ? lyzp[m0 + threadIdx.x] : 1e30f;
}

// accumulator row i, NT columns m, divided by lam_x,i + s_l[m] -> data operand (n = m, k = i)
template <int NW>
__device__ __forceinline__ void mid_scale(const Cta &c, int mtx, int NT, int nx, int px, const float *__restrict__ lx,
                                          const float *s_l, unsigned char *dsm, uint32_t off, uint32_t part) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nc = NT >> 4, k8 = px >> 3;
    for (int e = warp >> 2; e < mtx * nc; e += NW >> 2) {
        const int t = e / nc, cb = (e - t * nc) << 4;
        const int i = t * 128 + (warp & 3) * 32 + lane;
        float v[16];
        tmem_ld16(c.tmem + t * NT + cb + ((uint32_t)((warp & 3) * 32) << 16), v);
        const float li = i < nx ? lx[i] : 1e30f;
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = i < nx ? __fdividef(v[q], li + s_l[cb + q]) : 0.f;
        // even lanes store (i, i + 1) of column q, odd lanes (i - 1, i) of column q + 1
#pragma unroll
        for (int q = 0; q < 16; q += 2) {
            const float got = __shfl_xor_sync(0xffffffffu, (lane & 1) ? v[q] : v[q + 1], 1);
            const float x0 = (lane & 1) ? got : v[q], x1 = (lane & 1) ? v[q + 1] : got;
            const bf h0 = __float2bfloat16(x0), h1 = __float2bfloat16(x1);
            const uint32_t o = off + coff<LBD>(cb + q + (lane & 1), i & ~1, k8);
            if (i < px) {
                *reinterpret_cast<uint32_t *>(dsm + o) = pack2(h0, h1);
                *reinterpret_cast<uint32_t *>(dsm + o + part) =
                    pack2(__float2bfloat16(x0 - __bfloat162float(h0)), __float2bfloat16(x1 - __bfloat162float(h1)));
            }
        }
    }
}

inline int pad16(int x) { return (x + 15) / 16 * 16; }
inline int tiles128(int x) { return (x + 127) / 128; }
inline int cols_of(int need) {                    // tensor-memory columns: a power of two >= 32
    int t = 32;
    while (t < need) t *= 2;
    return t;
}
inline uint32_t axis_bytes(int P) { return (uint32_t)tiles128(P) * 16 * (P >> 3) * LBA; }
inline uint32_t data_bytes(int N, int K) { return (uint32_t)(N >> 3) * (K >> 3) * LBD; }
// (y, z) columns of a middle tile: 64, or 32 where 64 would leave SMs without a tile
inline int mid_cols(int ncol) { return (ncol + 63) / 64 >= 120 ? 64 : 32; }

}  // namespace sepp
