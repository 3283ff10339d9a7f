// The float64 Grams X^T A and X^T B (Lambda0 = X^T H X, S = X^T B X; Sec. 4.1) on the tensor cores: the
// blocks as integer digits (digits.cuh), 36 digit products per contraction.
//
// What bounds it: the direct form (k_gram2, block.cu) issues ld float64 multiply-adds per entry of A and
// B on a pipe that takes 16 cycles for a warp's.  Here an entry of a block costs ~45 integer and float32
// instructions once, and every 64 rows each of the 2 ld^2 sums costs ~80 and one float64 addition:
// 4.53 -> 1.23 ms at n = 1.18 M, p = 41; 0.135 -> 0.082 at n = 68k, p = 23 (with the idle fallback).
//
// A CTA owns a tile pair (i, j) of nh columns each and a range of rows, and walks it 64 rows at a time.
// The contracted index is the row, so every column of the 64 has an exponent of its own; a thread takes
// eight rows of a column, lanes along the columns, and stores 16 bytes of each digit.  The columns of
// [A | B] are the accumulator's rows (2 nh <= 128) and the digits of X side by side its columns: digit t
// of [A | B] times digits 0 .. 7 - t of X, written t nh columns further right, adds each product to the
// sum of its weight 2^(8 (14 - s - t)) in one or two instructions.  The eight sums of an entry (exact:
// below 2^23) are combined in integers, rounded once and added in float64.  The next 64 rows are loaded
// meanwhile.  Per-CTA partials go to part in k_gram2's layout.  Every wait is bounded, as in grad_tc.cu.
//
// Accuracy, entry by entry: 64 rows are off by at most 64 x 8.04 2^-60 of the product of the two columns'
// largest magnitudes there (COARSE in units of 64 2^-53 of it), a direct sum of 64 rows by 64 2^-53 of their
// sum of magnitudes.  The sums of 64 rows that are at hand bound the latter from below, so each CTA also adds
// |sum| - COARSE x (the product of the largest) over its rows, the least of four columns for all of them.
// Where the total of these over all rows is less than GRAM_DIG_LEAST (columns that share few rows, or are
// zero), or values are infinite, subnormal or beyond 2^60, the flag that k_gram_fin sets has k_gram2 add all
// entries up in float64.  So no entry's bound is larger than that of direct sums of 64 rows.  The smooth blocks
// and the noise of the runs measured never set it; localized columns that do pay for both
// forms (2.24 ms at n = 442k, p = 41, columns decaying as exp(-1.5 r); the direct form alone 1.74).
#include <algorithm>

#include "digits.cuh"

namespace {

using namespace sepp;

constexpr int GK = 64, GTH = 384, GK8 = GK / 8;   // rows per step, threads
constexpr float COARSE = 0.064f;                  // 8.04 2^-60 / 2^-53, and the rounding of the slack itself

__device__ __forceinline__ void tmem_ld4(uint32_t addr, float *v) {
    uint32_t u[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3])
                 : "r"(addr));
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(u[i]);
}

// integer value of a float32 integer: by the bits up to 2^22, by conversion beyond
__device__ __forceinline__ int small_int(float v) { return __float_as_int(v + 12582912.f) - 0x4b400000; }

template <int NH>
__global__ void __launch_bounds__(GTH, NH <= 2 ? 2 : 1)
    k_gram_dig(int64_t n, int p, int ld, int ntile, int tcols, const double *__restrict__ X, const double *__restrict__ A,
               const double *__restrict__ B, double *part, float *slack, int *redo, int64_t rows_per_split, int *err) {
    constexpr int nh = 16 * NH, NC = 3 * nh;                        // columns of X, A and B of a step
    constexpr uint32_t AD = 2 * nh / 8 * GK8 * LBA, XD = nh / 8 * GK8 * LBA;   // bytes of a digit of [A | B], of X
    constexpr int DM = 256 / nh < dig::NB ? 256 / nh : dig::NB;     // digits of X per instruction
    constexpr int CH = (4 * NH + 2) / 3;                            // chunks of four accumulator columns per thread
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag, s_bad, sE[2][NC];
    // accumulator rows past 2 nh read past a digit of [A | B], at most into X's, and are not read back
    const uint32_t sA = su32(dsm), sX = sA + dig::NB * AD;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int pair = blockIdx.x, ti = 0;
    while (pair >= ntile - ti) { pair -= ntile - ti; ++ti; }
    const int i0 = ti * nh, j0 = (ti + pair) * nh;
    const int64_t r0 = blockIdx.y * rows_per_split, r1 = r0 + rows_per_split < n ? r0 + rows_per_split : n;
    for (int e = tid; e < 2 * NC; e += GTH) sE[e / NC][e % NC] = 0;
    if (tid == 0) s_bad = 0;
    if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) *redo = 0;
    Cta c;
    cta_open(c, &mbar, &tmem_base, &abort_flag, tcols);
    double x[NH][8], acc[CH][4];
    float over[CH];                                   // a lower bound of the slack of acc's four entries
#pragma unroll
    for (int k = 0; k < CH; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[k][j] = 0.0;
#pragma unroll
    for (int k = 0; k < CH; ++k) over[k] = 0.f;
    auto fetch = [&](int64_t rb) {
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const int q = tid + GTH * i, g = q / NC, cc = q % NC, m = cc / nh, col = (m == 0 ? i0 : j0) + cc % nh;
            const double *src = (m == 0 ? X : (m == 1 ? A : B)) + col;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int64_t row = rb + 8 * g + r;
                x[i][r] = col < ld && row < r1 ? src[row * ld] : 0.0;
            }
        }
    };
    if (r0 < r1) fetch(r0);
    int par = 0;
    for (int64_t rb = r0; rb < r1; rb += GK, par ^= 1) {
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            int mx = 0;
#pragma unroll
            for (int r = 0; r < 8; ++r) mx = max(mx, dig::exponent(x[i][r]));
            if (mx == 0)
#pragma unroll
                for (int r = 0; r < 8; ++r) mx |= dig::nonzero(x[i][r]) ? 1 : 0;
            if (mx) atomicMax(&sE[par][(tid + GTH * i) % NC], mx);
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const int q = tid + GTH * i, g = q / NC, cc = q % NC;
            const int e = sE[par][cc];
            if (e > 0 && (e < 128 || e > 1023 + 60)) s_bad = 1;
            const uint32_t dst = cc < nh ? sX + coff<LBA>(cc, 8 * g, GK8) : sA + coff<LBA>(cc - nh, 8 * g, GK8);
            const uint32_t step = cc < nh ? XD : AD;
            uint32_t hi[8], lo[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const unsigned long long w = dig::bytes_of(x[i][r], e);
                hi[r] = (uint32_t)(w >> 32);
                lo[r] = (uint32_t)w;
            }
#pragma unroll
            for (int s = 0; s < dig::NB; ++s) {
                uint32_t w[4];
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    w[h] = __byte_perm(dig::digit_of(s < 4 ? hi[2 * h] : lo[2 * h], 3 - (s & 3)),
                                       dig::digit_of(s < 4 ? hi[2 * h + 1] : lo[2 * h + 1], 3 - (s & 3)), 0x7632);
                st16(dst + s * step, make_uint4(w[0], w[1], w[2], w[3]));
            }
        }
        asm volatile("fence.proxy.async.shared::cta;");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (tid == 0) {
            for (int kk = 0; kk < GK / 16; ++kk)
                for (int t = 0; t < dig::NB; ++t)
                    for (int s = 0; s < dig::NB - t; s += DM) {
                        const int cnt = min(DM, dig::NB - t - s);
                        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(cnt * nh >> 3) << 17) | (8u << 24);
                        const uint64_t ad = sdesc(sA + t * AD + kk * 2 * LBA, LBA, GK8 * LBA);
                        const uint64_t bd = sdesc(sX + s * XD + kk * 2 * LBA, LBA, GK8 * LBA);
                        const uint32_t accum = (t > 0 || kk > 0) ? 1u : 0u;
                        asm volatile(
                            "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(c.tmem + (t + s) * nh),
                            "l"(ad), "l"(bd), "r"(idesc), "r"(accum));
                    }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(c.mbar));
        }
        if (tid < NC) sE[par ^ 1][tid] = 0;           // its last readers passed the barriers above
        if (rb + GK < r1) fetch(rb + GK);
        uint32_t done = 0;
        for (long long w = 0; w < WAIT && !done; ++w)
            asm volatile(
                "{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}\n"
                : "=r"(done)
                : "r"(c.mbar), "r"(c.phase & 1));
        c.phase++;
        if (!done) abort_flag = 1;
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (abort_flag) break;
        const int m = (warp & 3) * 32 + lane;         // column of [A | B]
        if ((warp & 3) * 32 < 2 * nh) {
            const int eA = sE[par][nh + m];
#pragma unroll
            for (int k = 0; k < CH; ++k) {
                const int cb = 4 * ((warp >> 2) + 3 * k);
                if (cb >= nh) break;
                float v[dig::NB][4];
#pragma unroll
                for (int d = 0; d < dig::NB; ++d)
                    tmem_ld4(c.tmem + ((uint32_t)((warp & 3) * 32) << 16) + d * nh + cb, v[d]);
                asm volatile("tcgen05.wait::ld.sync.aligned;");
                float least = INFINITY;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    // sum d has d + 1 digit products, two of them with a top digit of at most 65: pairs of
                    // sums fit 32 bits, and the first four are at most 2^22
                    const int a = (small_int(v[0][j]) << 8) + small_int(v[1][j]), b = (small_int(v[2][j]) << 8) + small_int(v[3][j]);
                    const int f = ((int)v[4][j] << 8) + (int)v[5][j], g = ((int)v[6][j] << 8) + (int)v[7][j];
                    const long long hi = ((long long)a << 16) + b, lo = ((long long)f << 16) + g;
                    const int eX = sE[par][cb + j];
                    acc[k][j] += dig::combine<32>(hi, lo, eX + eA - 2 * 1084 + 56);
                    // |sum| in units of the two largest (2^34 in hi), less COARSE, times these (zero below 2^-126)
                    const float of = fmaf(fabsf((float)(int)(hi >> 12)), 0x1p-22f, -COARSE) *
                                     __int_as_float(max(eX + eA - 1919, 0) << 23);
                    if (eX) least = fminf(least, of);              // a zero column's products are zero
                }
                over[k] += least;
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
    }
    cta_close(c, tcols, err);
    const int m = (warp & 3) * 32 + lane, mat = m / nh, jj = m % nh;
    if (m >= 2 * nh || j0 + jj >= p) return;
#pragma unroll
    for (int k = 0; k < CH; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int ii = 4 * ((warp >> 2) + 3 * k) + j;
            if (ii < nh && i0 + ii <= j0 + jj) {
                const int64_t at = ((((int64_t)blockIdx.x * 2 + mat) * nh + ii) * nh + jj) * gridDim.y + blockIdx.y;
                part[at] = acc[k][j];
                slack[at] = s_bad ? -INFINITY : over[k];
            }
        }
}

}  // namespace

// float64 Grams by digits into the per-split partials of k_gram_fin (tiles of f->ts columns, f->ntile per side,
// f->splits ranges of rows); false where the form does not apply (the caller then runs the CUDA-core kernel).
// f->slack and f->redo: see above.
bool launch_gram_dig(ofks_ctx *c, const double *X, const double *A, const double *B, double *part, GramDig *f) {
    const int p = c->p, ld = c->ld;
    if (ld < GRAM_DIG_MIN) return false;
    const int nt = (p + 63) / 64, NH = ((p + nt - 1) / nt + 15) / 16, nh = 16 * NH, npair = nt * (nt + 1) / 2;
    const int tcols = cols_of(dig::NB * nh);
    const int smem = dig::NB * (3 * nh / 8 * GK8 * LBA);
    const int64_t slabs = (c->n + GK - 1) / GK;
    const int64_t want = std::max<int64_t>(1, std::min<int64_t>(slabs, (NH <= 2 ? 304 : 152) / npair));
    const int64_t rps = (slabs + want - 1) / want * GK, splits = (c->n + rps - 1) / rps;
    const int64_t count = 2LL * npair * nh * nh * splits;           // float64 partials, and as many float32
    if (count + (count + 1) / 2 > c->cpart_cap) return false;
    f->ts = nh; f->ntile = nt; f->splits = splits;
    f->slack = reinterpret_cast<float *>(part + count);
    f->redo = c->d_flag + 3;
#define GO_(k) { cudaFuncSetAttribute(k_gram_dig<k>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); \
    k_gram_dig<k><<<dim3((unsigned)npair, (unsigned)splits), GTH, smem, c->stream>>>(c->n, p, ld, nt, tcols, X, A, B, part, \
                                                                                    f->slack, f->redo, rps, c->d_flag + 2); }
    switch (NH) { case 1: GO_(1) break; case 2: GO_(2) break; case 3: GO_(3) break; default: GO_(4) }
#undef GO_
    return true;
}
