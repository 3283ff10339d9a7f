// The Hartree CG's separable preconditioner in three kernels instead of eight (sep_plane.cuh): the
// forward pass takes the CG update with it (U, r, r.r), the backward pass writes z and sums r.z.
//
// What bounds it: the passes are short (the tensor pipe is nearly idle, a pass moves 10-60 MB
// through L2 on the 80x44x43 chain), so launches, barriers and the latency of the first loads are
// what is left: 0.080 ms per application on that chain against 0.135 for the six-pass form, its
// gather and its scatter (events around each).
#include <algorithm>

#include "sep_plane.cuh"

namespace {

using namespace sepp;

constexpr int NT_ = 256, NW_ = NT_ / 32;          // threads and warps per CTA

struct Plane {
    int nx, ny, nz, py, pz;                       // interior extents; rounded up to 16
    const bf *Sa, *Sb;                            // axis matrices of the first and the second contraction
    float *T;                                     // tensor between the passes, [a][j][pz]
    int late;                                     // the second axis matrix reuses the first one's room
    uint32_t oB, oA2, part;                       // shared-memory offsets: data, second axis; bytes per data part
    int tcols;
    int *err;
    Vecs V;                                       // the CG vectors, and its scalars
    double *pw;
    float2 *pf;
    double *sc;
    int it, slot;
    double *gpart;
    unsigned *gcount;
};

// Forward pass, plane a: T1[k][b] = sum_c Sz[c][k] r[b][c], T2[j][k] = sum_b Sy[b][j] T1[k][b].
// With it >= 0 the CG update of iteration it comes first (the scalars protocol of the Hartree CG
// in fields.cu): alpha = rz/pq, U += alpha p, r -= alpha q, rr' += r.r, and the next pq slot is
// cleared.
__global__ void __launch_bounds__(NT_, 2) k_plane_fwd(const Plane P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    __shared__ double sh[8], s_alpha;
    const uint32_t sm = su32(dsm), sB = sm + P.oB;
    const int mtz = (P.pz + 127) >> 7, mty = (P.py + 127) >> 7, a = blockIdx.x;
    if (threadIdx.x == 0) {
        s_alpha = 0.0;
        if (P.it >= 0) {
            const double rz = P.sc[P.it & 1], pq = P.sc[2 + (P.it & 1)];
            s_alpha = pq > 0.0 ? rz / pq : 0.0;
        }
    }
    load_axis<NW_>(sm, P.Sa, P.pz);
    if (!P.late) load_axis<NW_>(sm + P.oA2, P.Sb, P.py);
    Cta c;
    cta_open(c, &mbar, &tmem_base, &abort_flag, P.tcols);
    double rr = 0.0;
    if (P.it >= 0) residual_to_data<NW_, 1>(P.V, a, P.ny, P.nz, P.py, P.pz, s_alpha, 0.0, rr, dsm, P.oB, P.part);
    else residual_to_data<NW_, 0>(P.V, a, P.ny, P.nz, P.py, P.pz, 0.0, 0.0, rr, dsm, P.oB, P.part);
    if (contract(c, sm, sB, P.part, mtz, P.py, P.pz)) {
        if (P.late) load_axis<NW_>(sm, P.Sb, P.py);
        acc_to_data<NW_>(c, mtz, P.py, P.pz, sB, P.part);          // row k, columns b
        if (contract(c, P.late ? sm : sm + P.oA2, sB, P.part, mty, P.pz, P.py))
            acc_to_global<NW_>(c, mty, P.pz, P.ny, P.pz, P.T + (int64_t)a * P.ny * P.pz, P.pz);
    }
    cta_close(c, P.tcols, P.err);
    if (P.it >= 0) {
        if (threadIdx.x == 0 && blockIdx.x == 0) P.sc[2 + ((P.it + 1) & 1)] = 0.0;
        const double tot[1] = {block_sum(rr, sh)};
        grid_accumulate<1>(tot, P.gpart, P.gcount, [&](int, double v) { P.sc[4 + ((P.it + 1) & 1)] += v; });
    }
}

// Backward pass, plane a: D[b][k] = sum_j Sy[b][j] T[j][k], z[c][b] = sum_k Sz[c][k] D[b][k], r.z
__global__ void __launch_bounds__(NT_, 2) k_plane_bwd(const Plane P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    __shared__ double sh[8];
    const uint32_t sm = su32(dsm), sB = sm + P.oB;
    const int mtz = (P.pz + 127) >> 7, mty = (P.py + 127) >> 7, a = blockIdx.x;
    load_axis<NW_>(sm, P.Sa, P.py);
    if (!P.late) load_axis<NW_>(sm + P.oA2, P.Sb, P.pz);
    Cta c;
    cta_open(c, &mbar, &tmem_base, &abort_flag, P.tcols);
    double rz = 0.0;
    global_to_data<NW_>(P.T + (int64_t)a * P.ny * P.pz, P.pz, P.ny, P.pz, P.pz, P.py, sB, P.part);
    if (contract(c, sm, sB, P.part, mty, P.pz, P.py)) {
        if (P.late) load_axis<NW_>(sm, P.Sb, P.pz);
        acc_to_data<NW_>(c, mty, P.pz, P.py, sB, P.part);          // row b, columns k
        if (contract(c, P.late ? sm : sm + P.oA2, sB, P.part, mtz, P.py, P.pz))
            acc_to_z<NW_, 0>(c, mtz, P.V, a, P.ny, P.nz, P.py, nullptr, P.pw, P.pf, rz);
    }
    cta_close(c, P.tcols, P.err);
    const double tot[1] = {block_sum(rz, sh)};
    grid_accumulate<1>(tot, P.gpart, P.gcount, [&](int, double v) { P.sc[P.slot] += v; });
}

struct Middle {
    int nx, px, ncol, NT;                         // ncol: (y, z) columns (ny pz); NT per tile
    const bf *St, *S;                             // x-axis modes, transposed and not
    const float *lx, *lyzp;                       // eigenvalues; lyzp padded like the columns (1e30)
    float *T;                                     // [a][column], in place
    int late;
    uint32_t oB, oA2, part;
    int tcols;
    int *err;
};

// Middle pass, NT columns m: D[i][m] = sum_a Sx[a][i] T[a][m], scaled, T'[a][m] = sum_i Sx[a][i] D[i][m]
__global__ void __launch_bounds__(NT_, 2) k_plane_mid(const Middle P) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    __shared__ float s_l[64];
    const uint32_t sm = su32(dsm), sB = sm + P.oB;
    const int mtx = (P.px + 127) >> 7, m0 = blockIdx.x * P.NT;
    load_axis<NW_>(sm, P.St, P.px);
    if (!P.late) load_axis<NW_>(sm + P.oA2, P.S, P.px);
    Cta c;
    cta_open(c, &mbar, &tmem_base, &abort_flag, P.tcols);
    mid_scales(P.lyzp, m0, P.ncol, P.NT, s_l);
    global_to_data<NW_>(P.T + m0, P.ncol, P.nx, P.ncol - m0, P.NT, P.px, sB, P.part);
    if (contract(c, sm, sB, P.part, mtx, P.NT, P.px)) {
        if (P.late) load_axis<NW_>(sm, P.S, P.px);
        mid_scale<NW_>(c, mtx, P.NT, P.nx, P.px, P.lx, s_l, dsm, P.oB, P.part);
        if (contract(c, P.late ? sm : sm + P.oA2, sB, P.part, mtx, P.NT, P.px))
            acc_to_global<NW_>(c, mtx, P.NT, P.nx, P.ncol - m0, P.T + m0, P.ncol);
    }
    cta_close(c, P.tcols, P.err);
}

// Shared memory of a pass: first axis matrix, second one (in the first one's room when both do
// not fit), data parts.  0: does not fit.
template <class Args>
int place(Args &P, int K1, int K2, uint32_t data) {
    const uint32_t a1 = axis_bytes(K1), a2 = axis_bytes(K2), d = 2 * data;
    P.part = data;
    P.late = a1 + a2 + d > (uint32_t)SMEM_MAX;
    if (!P.late) { P.oA2 = a1; P.oB = a1 + a2; }
    else { P.oA2 = 0; P.oB = std::max(a1, a2); }
    const uint32_t need = P.oB + d;
    if (need > (uint32_t)SMEM_MAX || P.tcols > 512) return 0;
    // at least as much shared memory as keeps more CTAs off an SM than its 512 tensor-memory
    // columns serve, so that no allocation waits
    return (int)std::min<uint32_t>(SMEM_MAX, std::max<uint32_t>(need, 228 * 1024 / (512 / P.tcols + 1) + 512));
}

int place_mid(const SepState &S, Middle &M) {
    M = Middle{};
    M.nx = S.n[0]; M.px = pad16(S.n[0]); M.ncol = S.n[1] * pad16(S.n[2]); M.NT = mid_cols(M.ncol);
    M.St = S.hSt[0]; M.S = S.hS[0]; M.lx = S.lx; M.lyzp = S.lyzp; M.T = S.t0;
    M.tcols = cols_of(tiles128(M.px) * M.NT);
    return place(M, M.px, M.px, data_bytes(M.NT, M.px));
}

int place_plane(const SepState &S, Plane &P, bool fwd) {
    P = Plane{};
    P.nx = S.n[0]; P.ny = S.n[1]; P.nz = S.n[2]; P.py = pad16(S.n[1]); P.pz = pad16(S.n[2]);
    P.T = S.t0;
    P.tcols = cols_of(std::max(tiles128(P.pz) * P.py, tiles128(P.py) * P.pz));
    P.Sa = fwd ? S.hSt[2] : S.hS[1];
    P.Sb = fwd ? S.hSt[1] : S.hS[2];
    return place(P, fwd ? P.pz : P.py, fwd ? P.py : P.pz, data_bytes(P.py, P.pz));
}

template <class K, class Args>
void go(ofks_ctx *c, K kern, Args &P, int items, int smem) {
    P.err = c->d_flag + 1;
    ofks_allow_smem((const void *)kern);
    kern<<<(unsigned)items, NT_, smem, c->stream>>>(P);
    c->kernels += 1;
}

}  // namespace

// the three-pass form applies: every pass's operands fit in shared and tensor memory (axes up to
// about 176 interior points; beyond, the six passes of separable.cu)
bool sep_plane_fits(const SepState &S) {
    Plane P;
    Middle M;
    return place_plane(S, P, true) && place_plane(S, P, false) && place_mid(S, M);
}

// Hartree CG: update of iteration it (it >= 0), z = A_sep^-1 r, rz[slot] += r.z; first: also p = z
void sep_plane_hartree(ofks_ctx *c, int it, int slot, int first) {
    const SepState &S = c->sep;
    Plane P;
    Middle M;
    auto vectors = [&]() {
        P.V = {c->st.Ly, c->st.Lz, c->d_cp, c->d_cq, c->d_U, c->d_cr, c->d_cz, nullptr};
        P.pw = first ? c->d_cp : nullptr; P.pf = first && c->hartree_ff ? c->d_cpff : nullptr;
        P.sc = c->d_sc + SC_CG; P.it = it; P.slot = slot; P.gpart = c->d_gpart; P.gcount = c->d_gcount;
    };
    int smem = place_plane(S, P, true);
    vectors();
    go(c, k_plane_fwd, P, S.n[0], smem);
    smem = place_mid(S, M);
    go(c, k_plane_mid, M, (M.ncol + M.NT - 1) / M.NT, smem);
    smem = place_plane(S, P, false);
    vectors();
    go(c, k_plane_bwd, P, S.n[0], smem);
}
