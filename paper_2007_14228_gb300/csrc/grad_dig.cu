// The float64 gradient G = H X + B X C and the residual norm |H X - B X Lambda0|_F (Alg. 2, Sec. 4.1)
// on the tensor cores: B X and [C | Lambda0] without their diagonals as integer digits (digits.cuh), 28
// digit products per contraction; the diagonals' terms are one float64 multiply-add each.
//
// What bounds it: the direct form issues 2 ld float64 multiply-adds per entry on a pipe that takes 16
// cycles for a warp's, 84 % of that pipe's peak; here an entry takes five float64 operations, and the
// rest is integer work on the digits (80 instructions per entry of B X, ~65 per output) and the
// readback of eight accumulators: 7.51 -> 1.89 ms at n = 1.18 M, p = 41; 2.83 -> 0.73 at n = 442k;
// 0.164 -> 0.099 at n = 68k, p = 23.
//
// Accuracy, entry by entry: the digits are off by at most 7.2 p 2^-59 of the product of the row's largest
// magnitude and the column's largest off the diagonal, the direct form's p multiply-adds by p 2^-53 of
// sum_k |B X_rk| |C_kc|.  A twenty-ninth product, of the magnitudes cut to eight bits with the diagonal,
// bounds that sum from below; where it is less than 7.2/64 of the two largest (a row whose large entries
// meet small ones of C), and for rows or columns beyond the digits' range, the products are added up in
// float64.  So no entry's bound is larger than the direct form's.  The diagonal stays out because it is
// often far larger than the rest of its column (blocks close to eigenvectors, or noise: 3.6 ms at n = 442k,
// p = 41 with most entries added up, 0.73 so).  On smooth blocks and noise none to 1e-5 of the entries are
// added up, on columns that share few rows nearly all (3.76 ms there, columns decaying as exp(-1.5 r); the direct
// form alone 2.83).
//
// One persistent CTA per SM walks 128-row tiles.  Two threads per row load it, agree on its largest
// exponent and write its seven digits and magnitudes as K-major operands; one thread issues the products
// of B X with C, 8 accumulators of nh columns in tensor memory; every warp reads its 32 rows and half of
// the columns back, combines, adds H X and the diagonal's term and stores G; then the same with Lambda0
// for the norm.  The next tile's rows are loaded meanwhile.  Every wait is bounded, as in grad_tc.cu.
#include <algorithm>

#include "digits.cuh"

namespace {

using namespace sepp;

constexpr int OT = 128, OTH = 256;                // rows per tile, threads
constexpr int NS = dig::ND + 1;                   // operands of a block: its digits and its magnitudes
constexpr float FINE = 7.2f / 64.f;               // least sum of magnitudes for which the digits stand
// exponents that the digits stand for: no infinities, and no subnormal values, products or results
__device__ __forceinline__ bool usable(int e) { return e == 0 || (e >= 575 && e < 2047); }

__device__ __forceinline__ void tmem_ld8(uint32_t addr, float *v) {
    uint32_t u[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7])
                 : "r"(addr));
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(u[i]);
}

// NH = nh / 16: operand width nh (ld rounded up to 16), nh / 2 columns per thread of a row
template <int NH>
__global__ void __launch_bounds__(OTH, 1) k_grad_dig(int64_t n, int p, int ld, int tcols, const double *__restrict__ HX,
                                                     const double *__restrict__ BX, const double *__restrict__ C,
                                                     const double *__restrict__ L0, double *G, double *kkt2, int *err,
                                                     double *gpart, unsigned *gcount) {
    constexpr int nh = 16 * NH, HALF = nh / 2, k8 = nh / 8;
    constexpr uint32_t AB = OT / 8 * k8 * LBA, BB = nh / 8 * k8 * LBA;   // bytes of a digit of B X, of C
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag, sE[OT], sEC[2][nh];
    __shared__ float sLeast[2][nh];                   // per column, the least sum of magnitudes
    __shared__ double sDiag[2][nh];                   // the diagonals
    __shared__ double red[OTH / 32];
    constexpr int PX = nh + 2;                                     // pitch of sX: rows 16 bytes apart in the banks
    const uint32_t sA = su32(dsm), sB = sA + NS * AB;              // operands of B X; of C and Lambda0
    double *sX = reinterpret_cast<double *>(dsm + NS * AB + 2 * NS * BB);   // the tile of B X
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t ntile = (n + OT - 1) / OT;
    Cta c;
    cta_open(c, &mbar, &tmem_base, &abort_flag, tcols);
    // C and Lambda0: largest exponent of each column, then the digits as (n = column, k = row)
    for (int e = tid; e < 2 * nh; e += OTH) {
        const double *M = e < nh ? C : L0;
        const int col = e < nh ? e : e - nh;
        int mx = 0;
        if (col < p)
            for (int k = 0; k < p; ++k) {
                const double v = k == col ? 0.0 : M[(int64_t)k * ld + col];
                mx = max(mx, max(dig::exponent(v), dig::nonzero(v) ? 1 : 0));
            }
        sEC[e < nh ? 0 : 1][col] = mx;
        sDiag[e < nh ? 0 : 1][col] = col < p ? M[(int64_t)col * ld + col] : 0.0;
        sLeast[e < nh ? 0 : 1][col] = mx == 0 ? -1.f : usable(mx) ? FINE : INFINITY;
    }
    __syncthreads();
    for (int e = tid; e < 2 * nh * nh; e += OTH) {
        const int m = e / (nh * nh), k = (e - m * nh * nh) / nh, col = e % nh;
        const double *M = m == 0 ? C : L0;
        const double v = k < p && col < p ? M[(int64_t)k * ld + col] : 0.0;
        uint32_t q[dig::ND];
        dig::split(k != col ? v : 0.0, sEC[m][col], q);
#pragma unroll
        for (int s = 0; s < NS; ++s)
            *reinterpret_cast<uint16_t *>(dsm + NS * AB + (uint32_t)(m * NS + s) * BB + coff<LBA>(col, k, k8)) =
                (uint16_t)(s < dig::ND ? q[s] : dig::magnitude(v, sEC[m][col]));
    }
    const int crow = tid >> 1, ccol = (tid & 1) * HALF;             // this thread's part of a row to convert
    double x[HALF];
    auto fetch = [&](int64_t tile) {
        const int64_t r = tile * OT + crow;
#pragma unroll
        for (int j = 0; j < HALF; j += 2) {
            double2 v = make_double2(0.0, 0.0);
            if (r < n && ccol + j < ld) v = *reinterpret_cast<const double2 *>(BX + r * ld + ccol + j);
            x[j] = v.x; x[j + 1] = v.y;
        }
    };
    // products of the tile's digits with matrix m, the seven accumulators side by side, and of the magnitudes
    auto multiply = [&](int m) {
        asm volatile("fence.proxy.async.shared::cta;");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (tid == 0) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(nh >> 3) << 17) | (8u << 24);
            for (int d = 0; d < NS; ++d)
                for (int s = d < dig::ND ? 0 : d; s <= d; ++s)
                    for (int kk = 0; kk < NH; ++kk) {
                        const int t = d < dig::ND ? d - s : d;
                        const uint64_t ad = sdesc(sA + s * AB + kk * 2 * LBA, LBA, k8 * LBA);
                        const uint64_t bd = sdesc(sB + (uint32_t)(m * NS + t) * BB + kk * 2 * LBA, LBA, k8 * LBA);
                        const uint32_t accum = ((d < dig::ND && s > 0) || kk > 0) ? 1u : 0u;
                        asm volatile(
                            "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(c.tmem + d * nh),
                            "l"(ad), "l"(bd), "r"(idesc), "r"(accum));
                    }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(c.mbar));
        }
    };
    auto wait = [&]() -> bool {
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
        return abort_flag == 0;
    };
    double part = 0.0;
    const int row = (warp & 3) * 32 + lane, col0 = (warp >> 2) * HALF;   // this thread's outputs of a tile
    // the coarse columns of row r in float64, four at a time (rare; a warp's four columns cost what they do in
    // the direct form)
    auto direct = [&](int m, int64_t r, unsigned coarse) {
        const double *M = m == 0 ? C : L0;
#pragma unroll 1
        for (int q = 0; q < HALF && col0 + q < ld; q += 4) {
            if (!__any_sync(0xffffffffu, coarse >> q & 15u)) continue;
            double t[4] = {0.0, 0.0, 0.0, 0.0};
            for (int k = 0; k < p; ++k) {
                const double b = r < n ? BX[r * ld + k] : 0.0;
#pragma unroll
                for (int j = 0; j < 4; ++j) t[j] = fma(b, __ldg(M + (int64_t)k * ld + col0 + q + j), t[j]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int col = col0 + q + j;
                if (!(coarse >> (q + j) & 1u) || col >= p) continue;
                const double hx = HX[r * ld + col];
                if (m == 0) G[r * ld + col] = hx + t[j];
                else part = fma(hx - t[j], hx - t[j], part);
            }
        }
    };
    if (blockIdx.x < ntile) fetch(blockIdx.x);
    for (int64_t tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        int mx = 0;
#pragma unroll
        for (int j = 0; j < HALF; ++j) mx = max(mx, dig::exponent(x[j]));
        if (mx == 0)
#pragma unroll
            for (int j = 0; j < HALF; ++j) mx |= dig::nonzero(x[j]) ? 1 : 0;
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        if ((tid & 1) == 0) sE[crow] = mx;
#pragma unroll
        for (int j = 0; j < HALF; j += 2)
            *reinterpret_cast<double2 *>(sX + crow * PX + ccol + j) = make_double2(x[j], x[j + 1]);
#pragma unroll
        for (int g = 0; g < NH; ++g) {
            uint32_t w[NS][4];
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                uint32_t a[dig::ND], b[dig::ND];
                dig::split(x[8 * g + j], mx, a);
                dig::split(x[8 * g + j + 1], mx, b);
#pragma unroll
                for (int s = 0; s < dig::ND; ++s) w[s][j >> 1] = a[s] | (b[s] << 16);
                w[dig::ND][j >> 1] = dig::magnitude(x[8 * g + j], mx) | (dig::magnitude(x[8 * g + j + 1], mx) << 16);
            }
#pragma unroll
            for (int s = 0; s < NS; ++s)
                st16(sA + s * AB + coff<LBA>(crow, ccol + 8 * g, k8), make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]));
        }
        multiply(0);
        const int64_t r = tile * OT + row;
        double h[HALF];
#pragma unroll
        for (int j = 0; j < HALF; j += 2) {
            double2 v = make_double2(0.0, 0.0);
            if (r < n && col0 + j < ld) v = *reinterpret_cast<const double2 *>(HX + r * ld + col0 + j);
            h[j] = v.x; h[j + 1] = v.y;
        }
        const int eR = sE[row];                       // written before multiply's barrier
        const float lift = eR == 0 ? FINE : 0.f;      // a zero row's products are zero
        for (int m = 0; m < 2; ++m) {
            if (!wait()) break;
            if (m == 1 && tile + gridDim.x < ntile) fetch(tile + gridDim.x);
            unsigned coarse = usable(eR) ? 0u : ~0u;  // the thread's columns whose digits are too coarse
#pragma unroll
            for (int cb = 0; cb < HALF; cb += 8) {
                float v[NS][8];
#pragma unroll
                for (int d = 0; d < NS; ++d)
                    tmem_ld8(c.tmem + ((uint32_t)((warp & 3) * 32) << 16) + d * nh + col0 + cb, v[d]);
                asm volatile("tcgen05.wait::ld.sync.aligned;");
                double g[8], b[8];
                if (m == 0)
#pragma unroll
                    for (int j = 0; j < 8; j += 2) {
                        const double2 t = *reinterpret_cast<const double2 *>(sX + row * PX + col0 + cb + j);
                        b[j] = t.x; b[j + 1] = t.y;
                    }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    long long hi = 0, lo = 0;
#pragma unroll
                    for (int d = 0; d < 4; ++d) hi = (hi << 9) + (int)v[d][j];
#pragma unroll
                    for (int d = 4; d < dig::ND; ++d) lo = (lo << 9) + (int)v[d][j];
                    const int col = col0 + cb + j;
                    const double val = dig::combine<27>(hi, lo, eR + sEC[m][col] - 2 * 1083 + 54);
                    if (v[dig::ND][j] + lift < sLeast[m][col]) coarse |= 1u << (cb + j);
                    if (m == 0) {
                        g[j] = h[cb + j] + fma(b[j], sDiag[0][col], val);
                        h[cb + j] = fma(-b[j], sDiag[1][col], h[cb + j]);
                    } else if (col < p && r < n && !(coarse >> (cb + j) & 1u)) {
                        const double res = h[cb + j] - val;
                        part = fma(res, res, part);
                    }
                }
                if (m == 0 && r < n)
#pragma unroll
                    for (int j = 0; j < 8; j += 2)
                        if (col0 + cb + j < ld)
                            *reinterpret_cast<double2 *>(G + r * ld + col0 + cb + j) = make_double2(g[j], g[j + 1]);
            }
            if (r >= n) coarse = 0u;
            if (__any_sync(0xffffffffu, coarse != 0u)) direct(m, r, coarse);
            if (m == 0) multiply(1);                  // its barrier follows the last read of the accumulators
        }
        if (abort_flag) break;
        asm volatile("tcgen05.fence::before_thread_sync;");
    }
    const double tot[1] = {block_sum(part, red)};
    cta_close(c, tcols, err);
    grid_accumulate<1>(tot, gpart, gcount, [&](int, double v) { *kkt2 += v; });
}

}  // namespace

// float64 gradient by digits; false where the form does not apply (the caller then runs the CUDA-core
// kernel).  kkt2 must be zero on entry.
bool launch_grad_dig(ofks_ctx *c, const double *HX, const double *BX, double *G, double *kkt2) {
    const int ld = c->ld;
    if (ld % 4 || ld < GRAD_DIG_MIN || ld > 48) return false;
    const int NH = (ld + 15) / 16, nh = 16 * NH;
    const int tcols = cols_of(NS * nh);
    const uint32_t k8 = nh / 8, smem = NS * (OT / 8 * k8 * LBA) + 2 * NS * (nh / 8 * k8 * LBA) + 8 * OT * (nh + 2);
    const int64_t ntile = (c->n + OT - 1) / OT;
    const unsigned grid = (unsigned)std::min<int64_t>(ntile, 152);
    // tensor memory for one CTA per SM where it takes more than half of the columns
    const int sm = (int)std::max<uint32_t>(smem, 228 * 1024 / (512 / tcols + 1) + 512);
#define GO_(k) { cudaFuncSetAttribute(k_grad_dig<k>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm); \
    k_grad_dig<k><<<grid, OTH, sm, c->stream>>>(c->n, c->p, ld, tcols, HX, BX, c->d_C, c->d_L0, G, kkt2, c->d_flag + 2, \
                                               c->d_gpart, c->d_gcount); }
    if (NH == 1) GO_(1) else if (NH == 2) GO_(2) else GO_(3)
#undef GO_
    c->kernels += 1;
    return true;
}
