// Device-side pieces shared by the batched coarse cycle kernels (coarse_block.cu,
// coarse_cycle.cu): 16-bit packing and the MMA of the block products, neighbours,
// gates, and the push of an Arnoldi column into the FP64 least squares.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "batch.cuh"
#include "coarse_block.cuh"
#include "ks_dev.cuh"

namespace mg {
namespace cbdev {

constexpr int NDOF = 24;
constexpr int TILE_WORDS = 64;
constexpr int SITE_WORDS = 5 * 9 * TILE_WORDS;
constexpr int MAXI = MSMAX + 1;  // basis vectors of a cycle

template <bool F16>
__device__ __forceinline__ unsigned pk(float re, float im) {
    if constexpr (F16) {
        const __half2 h = __floats2half2_rn(re, im);
        return *reinterpret_cast<const unsigned*>(&h);
    } else {
        const __nv_bfloat162 h = __floats2bfloat162_rn(re, im);
        return *reinterpret_cast<const unsigned*>(&h);
    }
}
template <bool F16>
__device__ __forceinline__ float2 upk(unsigned u) {
    if constexpr (F16) return __half22float2(*reinterpret_cast<const __half2*>(&u));
    else return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u));
}
template <bool F16>
__device__ __forceinline__ void mma(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    if constexpr (F16)
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
            "{%0,%1,%2,%3};\n"
            : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
    else
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
            "{%0,%1,%2,%3};\n"
            : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ unsigned embed(unsigned w, int p) {
    return p ? __byte_perm(w, 0u, 0x1032) : (w ^ 0x80000000u);
}
// neighbour site in direction d (self, +x, -x, +t, -t), periodic; 32-bit index
// arithmetic (a coarse grid has far fewer than 2^31 sites)
__device__ __forceinline__ int nbr_of(int s, int d, int Nx, int Nt) {
    const int t = s / Nx, xx = s - t * Nx;
    switch (d) {
        case 0: return s;
        case 1: return (xx + 1 == Nx) ? s - xx : s + 1;
        case 2: return (xx == 0) ? s + Nx - 1 : s - 1;
        case 3: return (t + 1 == Nt) ? xx : s + Nx;
        default: return (t == 0) ? s + Nx * (Nt - 1) : s - Nx;
    }
}

// the bits of the tile's right-hand sides whose gate opens step jh
__device__ __forceinline__ unsigned gate_mask(const int* gate, int r0, int jh) {
    unsigned m = 0u;
#pragma unroll
    for (int q = 0; q < NB_TILE; ++q) m |= (__ldcg(gate + r0 + q) == jh ? 1u : 0u) << q;
    return m;
}

// the least squares of a tile's right-hand sides during a cycle (FP64): rotations, the
// rotated right-hand side, the tolerance and a column; the products of the column to push
struct CBPush {
    double rc[NB_TILE][MSMAX];
    double2 rs[NB_TILE][MSMAX];
    double2 g[NB_TILE][MSMAX + 1];
    double2 col[NB_TILE][MAXI + 1];
    double tol[NB_TILE];
    float2 h1[NB_TILE][MAXI];  // first-pass products
    float hn[NB_TILE];
};

// column jh of right-hand side l: h1 + h2 with subdiagonal hn
__device__ __forceinline__ void push_column_entries(CBPush& S, int l, int jh, const float2* h2, int i0, int is) {
    for (int i = i0; i <= jh; i += is)
        S.col[l][i] = make_double2((double)S.h1[l][i].x + (double)h2[i].x, (double)S.h1[l][i].y + (double)h2[i].y);
    if (i0 == 0) S.col[l][jh + 1] = make_double2((double)S.hn[l], 0.0);
}

// The column in S.col[l] into right-hand side r's least squares (the cycle kernels'
// push): rotated by the cycle's earlier rotations (kept in shared memory, so no step waits
// on a dependent global load), a new rotation, the rotated right-hand side, the residual
// estimate and the gates.  stop: the decision already made (1: converged, 0: not), or -1
// to make it from the residual estimate.
// The state in global memory receives what the cycle's finish reads (H, R, g,
// rotations, j, res, conv) without being read back.
__device__ __forceinline__ void push_cycle(const CBArgs& a, CBPush& S, int l, int r, int jh, int stop) {
    KState* ks = a.ks + r;
    double2* col = S.col[l];
    const double hn = col[jh + 1].x;
    double2* Hc = ks->H + KLD * jh;
    double2* Rc = ks->R + KLD * jh;
    for (int i = 0; i <= jh + 1; ++i) Hc[i] = col[i];
    for (int i = jh + 2; i < KLD; ++i) {
        Hc[i] = make_double2(0.0, 0.0);
        Rc[i] = make_double2(0.0, 0.0);
    }
    double2 p = col[0];
    for (int t = 0; t < jh; ++t) {
        double2 q = col[t + 1];
        ksd::rot_apply(S.rc[l][t], S.rs[l][t], p, q);
        Rc[t] = p;
        p = q;
    }
    double cc;
    double2 ss, rr;
    ksd::givens(p, col[jh + 1], cc, ss, rr);
    Rc[jh] = rr;
    Rc[jh + 1] = make_double2(0.0, 0.0);
    S.rc[l][jh] = cc;
    S.rs[l][jh] = ss;
    ks->rc[jh] = cc;
    ks->rs[jh] = ss;
    ks->ra[jh] = (short)jh;
    ks->rb[jh] = (short)(jh + 1);
    ksd::rot_apply(cc, ss, S.g[l][jh], S.g[l][jh + 1]);
    ks->g[jh] = S.g[l][jh];
    ks->g[jh + 1] = S.g[l][jh + 1];
    const double res = ksd::cabsd(S.g[l][jh + 1]);
    const int conv = stop >= 0 ? stop : res <= S.tol[l] ? 1 : 0, brk = hn == 0.0 ? 1 : 0;
    const int next = (conv || brk || jh + 1 >= KMAX) ? -1 : jh + 1;
    ks->nrot = jh + 1;
    ks->res = res;
    ks->j = jh + 1;
    ks->conv = conv;
    ks->breakdown = brk;
    ks->step_gate = next;
    ks->scale_gate = hn > 0.0 ? jh + 1 : -1;
    ks->scale = hn > 0.0 ? 1.0 / hn : 0.0;
    a.gbuf[((jh + 1) & 1) * a.nbp + r] = next;
}

}  // namespace cbdev
}  // namespace mg
