// Device-side pieces of the Krylov least squares shared by the kernels that
// update it (dense.cu, and the fused coarse block steps in coarse_block.cu):
// complex Givens rotations and the incremental push of one Arnoldi column.
#pragma once
#include "kstate.cuh"

namespace mg {
namespace ksd {

__device__ __forceinline__ double cabsd(double2 a) { return sqrt(a.x * a.x + a.y * a.y); }
__device__ __forceinline__ double cabs2d(double2 a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ double cabs1d(double2 a) { return fabs(a.x) + fabs(a.y); }
// a / b = a conj(b) / |b|^2 with one real reciprocal: FP64 divides and square
// roots are long dependent sequences at this GPU's FP64 rate, and these sit on
// serial paths.  (The entries here are O(1e-16..1e2), far from overflow.)
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
    const double inv = 1.0 / cabs2d(b);
    return make_double2((a.x * b.x + a.y * b.y) * inv, (a.y * b.x - a.x * b.y) * inv);
}
__device__ __forceinline__ double2 z0() { return make_double2(0.0, 0.0); }

// Complex Givens rotation G = [[c, s], [-conj(s), c]] with G [a; b] = [r; 0].
// (reciprocal square roots only, no divide)
__device__ __forceinline__ void givens(double2 a, double2 b, double& c, double2& s, double2& r) {
    const double ab2 = cabs2d(b);
    if (ab2 == 0.0) {
        c = 1.0;
        s = z0();
        r = a;
        return;
    }
    const double aa2 = cabs2d(a);
    if (aa2 == 0.0) {
        const double inv_ab = rsqrt(ab2);
        c = 0.0;
        s = make_double2(b.x * inv_ab, -b.y * inv_ab);
        r = make_double2(ab2 * inv_ab, 0.0);
        return;
    }
    const double rho2 = aa2 + ab2;
    const double inv_aa = rsqrt(aa2), inv_rho = rsqrt(rho2);
    c = aa2 * inv_aa * inv_rho;
    const double2 ph = make_double2(a.x * inv_aa, a.y * inv_aa);
    s = cscale(cmul(ph, conj_(b)), inv_rho);
    r = cscale(ph, rho2 * inv_rho);
}
__device__ __forceinline__ void rot_apply(double c, double2 s, double2& up, double2& uq) {
    const double2 p = up, q = uq;
    up = cadd(cscale(p, c), cmul(s, q));
    uq = csub(cscale(q, c), cmul(conj_(s), p));
}

// Column jh of the Arnoldi matrix from hA + hB and sqrt(hn2): store it, apply the
// earlier rotations, add the new one, update the rotated right-hand side, the
// residual estimate, the stop flags and the gates of the next step.
__device__ inline void ks_push_dev(KState* ks, int jh) {
    if (ks->step_gate != jh) return;
    const int j = jh;
    double2* Hc = ks->H + KLD * j;
    double2* Rc = ks->R + KLD * j;
    for (int i = 0; i <= j; ++i) {
        const double2 h = cadd(ks->hA[i], ks->hB[i]);
        Hc[i] = h;
        Rc[i] = h;
    }
    for (int i = j + 2; i < KLD; ++i) {
        Hc[i] = z0();
        Rc[i] = z0();
    }
    const double hn = sqrt(fmax(ks->hn2, 0.0));
    Hc[j + 1] = make_double2(hn, 0.0);
    Rc[j + 1] = Hc[j + 1];
    const int nr = ks->nrot;
    for (int t = 0; t < nr; ++t) rot_apply(ks->rc[t], ks->rs[t], Rc[ks->ra[t]], Rc[ks->rb[t]]);
    double c;
    double2 s, r;
    givens(Rc[j], Rc[j + 1], c, s, r);
    Rc[j] = r;
    Rc[j + 1] = z0();
    ks->rc[nr] = c;
    ks->rs[nr] = s;
    ks->ra[nr] = (short)j;
    ks->rb[nr] = (short)(j + 1);
    ks->nrot = nr + 1;
    rot_apply(c, s, ks->g[j], ks->g[j + 1]);
    ks->res = cabsd(ks->g[j + 1]);
    ks->j = j + 1;
    ks->breakdown = (hn == 0.0) ? 1 : 0;
    ks->conv = (ks->res <= ks->tol_abs) ? 1 : 0;
    ks->step_gate = (ks->conv || ks->breakdown || j + 1 >= KMAX) ? -1 : j + 1;
    ks->scale_gate = (hn > 0.0) ? j + 1 : -1;
    ks->scale = (hn > 0.0) ? 1.0 / hn : 0.0;
}


// Start of a cycle from a vector of squared norm nrm2v, by one warp
__device__ inline void ks_start_dev(KState* ks, double nrm2v, double tol_rel, double nb2v) {
    const double beta = sqrt(fmax(nrm2v, 0.0));
    const double tol_abs = tol_rel * sqrt(fmax(nb2v, 0.0));
    const int lane = threadIdx.x & 31;  // one warp: lane 0 writes the scalars
    for (int i = lane; i < KLD; i += 32) ks->c[i] = ks->g[i] = make_double2(i == 0 ? beta : 0.0, 0.0);
    if (lane != 0) return;
    ks->beta = beta;
    ks->tol_abs = tol_abs;
    ks->res = beta;
    ks->nrot = 0;
    ks->j = 0;
    ks->j0 = 0;
    ks->conv = (beta <= tol_abs) ? 1 : 0;
    ks->breakdown = 0;
    ks->err = 0;
    ks->step_gate = (!ks->conv && beta > 0.0) ? 0 : -1;
    ks->scale = beta > 0.0 ? 1.0 / beta : 0.0;
    ks->scale_gate = 0;
}
// ks_push_dev by one warp: the column and the earlier rotations are read
// into shared memory at once, so that the serial chain of rotations (lane 0) waits for
// no dependent global load, and the column's zeros are written by all lanes.
struct PushScratch {
    double2 col[KLD];
    double2 rs[NROT];
    double rc[NROT];
    short ra[NROT], rb[NROT];
};
__device__ inline void ks_push_warp(KState* ks, int jh, PushScratch& S) {
    double2 *col = S.col, *rs = S.rs;
    double* rc = S.rc;
    short *ra = S.ra, *rb = S.rb;
    const int lane = threadIdx.x & 31, j = jh;
    if (ks->step_gate != jh) return;
    const int nr = ks->nrot;
    for (int t = lane; t < nr; t += 32) {
        rc[t] = ks->rc[t];
        rs[t] = ks->rs[t];
        ra[t] = ks->ra[t];
        rb[t] = ks->rb[t];
    }
    for (int i = lane; i <= j; i += 32) col[i] = cadd(ks->hA[i], ks->hB[i]);
    for (int i = j + 2 + lane; i < KLD; i += 32) col[i] = z0();
    const double hn2 = fmax(ks->hn2, 0.0), hn = sqrt(hn2), inv = hn > 0.0 ? 1.0 / hn : 0.0;
    if (lane == 0) col[j + 1] = make_double2(hn, 0.0);
    const double2 gj = ks->g[j];
    const double tol_abs = ks->tol_abs;
    __syncwarp();
    for (int i = lane; i < KLD; i += 32) ks->H[i + KLD * j] = col[i];
    __syncwarp();
    if (lane == 0) {
        for (int t = 0; t < nr; ++t) rot_apply(rc[t], rs[t], col[ra[t]], col[rb[t]]);
        double c;
        double2 sn, r;
        givens(col[j], col[j + 1], c, sn, r);
        col[j] = r;
        col[j + 1] = z0();
        ks->rc[nr] = c;
        ks->rs[nr] = sn;
        ks->ra[nr] = (short)j;
        ks->rb[nr] = (short)(j + 1);
        ks->nrot = nr + 1;
        double2 g0 = gj, g1 = ks->g[j + 1];
        rot_apply(c, sn, g0, g1);
        ks->g[j] = g0;
        ks->g[j + 1] = g1;
        const double res = cabsd(g1);
        const int conv = res <= tol_abs ? 1 : 0, brk = hn == 0.0 ? 1 : 0;
        ks->res = res;
        ks->j = j + 1;
        ks->breakdown = brk;
        ks->conv = conv;
        ks->step_gate = (conv || brk || j + 1 >= KMAX) ? -1 : j + 1;
        ks->scale_gate = (hn > 0.0) ? j + 1 : -1;
        ks->scale = inv;
    }
    __syncwarp();
    for (int i = lane; i < KLD; i += 32) ks->R[i + KLD * j] = col[i];
}
// Columns 0..jj - 1 of the upper triangle R, column i's rows 0..i at i (i + 1) / 2, by nt
// threads: several loads of a thread are in flight (a loop over columns waited for each)
__device__ __forceinline__ void load_upper(double2* Rs, const double2* R, int jj, int tid, int nt) {
#pragma unroll 4
    for (int e = tid; e < jj * jj; e += nt) {
        const int i = e / jj, r = e - i * jj;
        if (r <= i) Rs[i * (i + 1) / 2 + r] = R[r + KLD * i];
    }
}
// Back substitution R d = g over the first jj < 64 columns, by one warp: the lanes form the
// reciprocals of their pivots together (a zero pivot gives d_i = 0 and *err = 2), and each
// column then costs a product, a broadcast and a subtraction on the serial chain.
__device__ inline void solve_upper(const double2* Rs, const double2* g, double2* d, int jj, int* err) {
    const int lane = threadIdx.x & 31;
    double2 acc[2], inv[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int r = lane + 32 * h;
        acc[h] = inv[h] = z0();
        if (r < jj) {
            acc[h] = g[r];
            const double2 piv = Rs[r * (r + 1) / 2 + r];
            if (piv.x == 0.0 && piv.y == 0.0) {
                if (err) *err = 2;
            } else {
                inv[h] = cdiv(make_double2(1.0, 0.0), piv);
            }
        }
    }
    for (int i = jj - 1; i >= 0; --i) {
        const double2* Ri = Rs + i * (i + 1) / 2;
        double2 di = i >= 32 ? cmul(acc[1], inv[1]) : cmul(acc[0], inv[0]);
        di.x = __shfl_sync(0xffffffffu, di.x, i & 31);
        di.y = __shfl_sync(0xffffffffu, di.y, i & 31);
        if (lane == (i & 31)) d[i] = di;
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (lane + 32 * h < i) acc[h] = csub(acc[h], cmul(Ri[lane + 32 * h], di));
    }
    __syncwarp();
}

}  // namespace ksd
}  // namespace mg
