// Device pieces shared by the thread-block-cluster kernels of the coarsest-grid
// GMRES-Proj (coarse_coop.cu, coarse_tc.cu): the small least squares of a cycle,
// the dataflow exchange (st.async counted on mbarriers), bounded waits, and the
// neighbour geometry.
#pragma once
#include "coarse_coop.cuh"

namespace mg {
namespace cdev {

constexpr int NDOF = 24;
constexpr int MAX_CLUSTER = 16;       // CTAs of one cluster (non-portable size)
constexpr size_t SMEM_LIMIT = 227 * 1024;
constexpr long FLOW_SPIN = 1L << 20;  // default try_wait rounds before a dataflow wait gives up

template <typename R>
struct Small {  // per-CTA copy of the small least-squares state, precision R
    using Z = C2<R>;
    Z H[(MSMAX + 1) * MSMAX];  // column-major, ld MSMAX + 1 (unrotated)
    Z Rm[(MSMAX + 1) * MSMAX];
    R rc[MSMAX];
    Z rs[MSMAX];
    Z g[MSMAX + 1], c[MSMAX + 1];
    // coefficients of the row updates (read 16 bytes at a time)
    alignas(16) Z d[MSMAX];
    alignas(16) Z rho[MSMAX + 1];
    alignas(16) Z pd[KMAX];    // projection coefficients
    alignas(16) Z pu[KLD];
};

template <typename R>
__device__ __forceinline__ R cabs_(C2<R> a) { return sqrt(a.x * a.x + a.y * a.y); }

template <typename R>
__device__ __forceinline__ C2<R> cdiv_(C2<R> a, C2<R> b) {
    if (fabs(b.x) >= fabs(b.y)) {
        R r = b.y / b.x, den = b.x + b.y * r;
        return mk<R>((a.x + a.y * r) / den, (a.y - a.x * r) / den);
    }
    R r = b.x / b.y, den = b.x * r + b.y;
    return mk<R>((a.x * r + a.y) / den, (a.y * r - a.x) / den);
}

// acc - a * b with every rounding step fixed: both cluster kernels get the same
// operations, whatever contraction the compiler would pick for a * b - c * d
template <typename R>
__device__ __forceinline__ C2<R> cfms_(C2<R> a, C2<R> b, C2<R> acc) {
    acc.x = fma(-a.x, b.x, acc.x);
    acc.x = fma(a.y, b.y, acc.x);
    acc.y = fma(-a.x, b.y, acc.y);
    acc.y = fma(-a.y, b.x, acc.y);
    return acc;
}

// d = R^{-1} g for the jc x jc upper-triangular R (column-major, leading
// dimension MSMAX + 1, jc <= MSMAX < 32) by one warp, column by column. The
// lanes first form the reciprocals of their pivots at once (a zero pivot gives
// zero, so d_i = 0 there); then lane i keeps g_i minus the columns already
// eliminated, and in turn i its d_i = (that) / R_ii is broadcast to the lanes
// above.  Only a product, a shuffle and a subtraction stay on the serial chain.
template <typename R>
__device__ __forceinline__ void back_subst_warp(const C2<R>* Rm, const C2<R>* g, C2<R>* d, int jc, int lane) {
    constexpr int LDR = MSMAX + 1;
    C2<R> inv = mk<R>(0, 0), acc = mk<R>(0, 0);
    if (lane < jc) {
        const C2<R> piv = Rm[lane + LDR * lane];
        if (piv.x != R(0) || piv.y != R(0)) inv = cdiv_<R>(mk<R>(1, 0), piv);
        acc = g[lane];
    }
    for (int i = jc - 1; i >= 0; --i) {
        const C2<R> rli = (lane < i) ? Rm[lane + LDR * i] : mk<R>(0, 0);
        C2<R> di = mk<R>(fma(-acc.y, inv.y, acc.x * inv.x), fma(acc.y, inv.x, acc.x * inv.y));
        di.x = __shfl_sync(0xffffffffu, di.x, i);
        di.y = __shfl_sync(0xffffffffu, di.y, i);
        if (lane == i) d[i] = di;
        if (lane < i) acc = cfms_<R>(rli, di, acc);
    }
}

template <typename R>
__device__ __forceinline__ R rsqrt_(R x) {
    if constexpr (std::is_same<R, float>::value)
        return rsqrtf(x);
    else
        return rsqrt(x);
}

// Complex Givens rotation G = [[c, s], [-conj(s), c]] with G [a; h] = [r; 0]
// for a real, non-negative h (the new subdiagonal entry).
template <typename R>
__device__ __forceinline__ void givens_real_(C2<R> a, R h, R& c, C2<R>& s, C2<R>& r) {
    if (h == R(0)) { c = R(1); s = mk<R>(0, 0); r = a; return; }
    const R aa2 = a.x * a.x + a.y * a.y;
    if (aa2 == R(0)) { c = R(0); s = mk<R>(1, 0); r = mk<R>(h, 0); return; }
    // reciprocal square roots only: no divide on this serial path
    const R rh2 = aa2 + h * h;
    const R inv_aa = rsqrt_(aa2), inv_rh = rsqrt_(rh2);
    c = aa2 * inv_aa * inv_rh;
    const C2<R> ph = mk<R>(a.x * inv_aa, a.y * inv_aa);
    s = cscale(ph, h * inv_rh);
    r = cscale(ph, rh2 * inv_rh);
}
template <typename R>
__device__ __forceinline__ void rot_(R c, C2<R> s, C2<R>& up, C2<R>& uq) {
    const C2<R> p = up, q = uq;
    up = cadd(cscale(p, c), cmul(s, q));
    uq = csub(cscale(q, c), cmul(conj_(s), p));
}

// Split cluster barrier: arrive (releasing this thread's writes, shared and
// global, to the cluster) and wait (acquiring everyone's).  Work placed between
// the two overlaps the barrier's latency.  Every thread of a warp executes both.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }

// Dataflow exchange (push mode): instead of a cluster barrier after each push,
// every value goes out by st.async, which counts its bytes on an mbarrier in the
// receiving CTA; a CTA goes on once its barrier has seen all the bytes of the
// phase (armed by its thread 0 with the expected count).
__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned cluster_addr(unsigned local, int rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arm(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
// bounded wait for the completion of the phase with this parity (acquiring the
// cluster's st.async writes); false when it gave up
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, long spin) {
    const unsigned addr = smem_addr(bar);
    for (long it = 0; it < spin; ++it) {
        unsigned ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(addr), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}
// barrier 1 over the first nthreads threads (the row warps)
__device__ __forceinline__ void row_warps_sync(int nthreads) {
    asm volatile("bar.sync 1, %0;\n" ::"r"(nthreads) : "memory");
}
__device__ __forceinline__ void st_async(unsigned dst, float2 v, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];\n" ::"r"(dst),
                 "f"(v.x), "f"(v.y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_async(unsigned dst, double2 v, unsigned bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];\n" ::"r"(dst),
                 "d"(v.x), "d"(v.y), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ long nbr_site(long s, int d, int Nx, int Nt) {
    const int xx = (int)(s % Nx), tt = (int)(s / Nx);
    if (d == 1) return (xx + 1 == Nx) ? s - xx : s + 1;
    if (d == 2) return (xx == 0) ? s + Nx - 1 : s - 1;
    if (d == 3) return (tt + 1 == Nt) ? (long)xx : s + Nx;
    if (d == 4) return (tt == 0) ? s + (long)Nx * (Nt - 1) : s - Nx;
    return s;
}

}  // namespace cdev
}  // namespace mg
