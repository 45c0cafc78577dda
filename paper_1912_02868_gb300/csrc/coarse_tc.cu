// The mixed-precision coarsest-grid GMRES-Proj (Section 2; Morgan & Wilcox) as one
// thread-block-cluster kernel with its operator and basis on chip: FP32 vectors,
// FP16 operator applied on tensor cores, CGS2, at most 16 coarse sites a CTA.
// The method, the exchanges and the bounded waits are those of coarse_coop.cu,
// which serves every other case (FP64, FP32 operator or FMAs, delayed CGS2,
// larger slices).
//
// A step is a chain of latencies, not of bytes, so each link is cut short:
//  * Operator.  Warp w owns site w.  Its A fragments stay on chip for the whole
//    solve, half in the warp's registers and half in shared memory in fragment
//    order (one 16- and one 8-byte load a K tile), so the apply reads nothing
//    from L2.
//  * Vectors.  A basis row is staged once as the B fragment words themselves
//    (two FP16 parts, both real-form columns), so an apply's operand is one
//    8-byte load with no conversion.  A CTA's own rows are written locally; only
//    rows a neighbouring CTA reads travel, 16 bytes per st.async.
//  * Inner products.  A warp forms two products at once over the CTA's rows, so w is
//    read once for both; the partials go into inbox rows an odd number of 16-byte pairs
//    apart (no bank conflicts).
//  * The residual and the solution live on chip, the deflation space too when it
//    fits; every exchange is dataflow, and the per-cycle cluster barrier (which only
//    publishes faults) is split around the first one.
//
// Grid form (GRID): coarse grids of more than one cluster's 256 sites run on one
// cooperative grid over the whole GPU, a few sites a CTA.  An exchange then goes
// through L2 without barrier or fence: every 4-byte value is stored with a 4-byte
// tag of its exchange in one 8-byte word, and a reader polls the words themselves,
// so a value costs one store and, once it is there, one load.  Two buffers by the
// exchange's parity suffice: a CTA sends exchange e + 2 only after it has read e + 1,
// which holds every CTA's contribution, made after that CTA had read e.  Each
// projection exchange carries the CTAs' faults, so all leave together.
#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "coarse_dev.cuh"

namespace mg {

using namespace cdev;

namespace {

// Where a site's operator fragments sit: of a K tile, M tile 0 (rows 0..15) is four
// words a lane and M tile 1 (rows 16..23) two.  Registers hold M tile 0 of directions
// SD..4 and M tile 1 of directions SD1..4 (42 words: with 54 the loop spilled, and
// local memory misses the little L1 that the shared memory leaves).
constexpr int SD = 2, SD1 = 4;
constexpr int MAX_SITES = 16;
constexpr int XW = 48;      // words of one staged site: 12 entry pairs x (hi, hi, lo, lo)
constexpr int OPA = SD * 3 * 32, OPB = SD1 * 3 * 32;  // fragments of one site in shared memory, by M tile

// FP16 split of a staged value: hi = x 2^10 rounded to FP16, lo = the remainder times 2^11.
// The entries of a unit vector stay a factor 64 below the FP16 range, and lo is as large
// as hi, so that hi + 2^-11 lo carries 22 bits of entries down to 2^-24 (of a remainder on
// hi's own scale, entries below 2^-13 lose bits).  The products of the two parts are summed
// apart and scaled then.  Relative error of A v against 64 bits on the same FP16 operator,
// for Krylov and point-source vectors of 64^2 to 512^2 lattices: 2.4e-7 to 2.8e-7, where
// FP32 FMAs on the FP32 vector have 3.3e-7 to 3.7e-7 (one chain of 240 rounded sums).
constexpr float TC_XS = 1024.f;
constexpr float TC_RS = 2048.f;
constexpr float TC_XS_INV = 1.f / 1024.f;
constexpr float TC_XRS_INV = 1.f / (1024.f * 2048.f);

struct TcShape {
    int spc, halo, pw, ws, vrows;
    // byte offsets in dynamic shared memory
    int o_inbox, o_x, o_v, o_m, o_op, o_sol, o_w;
    // GRID: tagged partial sums [2][PSTR][CTAs], tagged rows [2][sites x 24], and the tag
    // base of this launch (advanced at its end) with a word that nothing writes (the probe's)
    ulonglong2 *part, *rows;
    unsigned* epoch;
};

struct alignas(16) TcSmem {
    // reduced products of the two exchange buffers, each as (x, y, y, x) for the packed
    // row updates, zero up to the next multiple of four; the norm apart
    float4 red[2][64];
    float nrm[2];
    alignas(16) float4 coef[2][64];  // coefficients of the cycle's row updates, the same way
    float2 u_ls[32], g_ls;           // least squares: the running row and right-hand-side entry
    int iters;
    alignas(16) int push[MAX_SITES][4];  // where own rows go: (CTA << 16) | slot, -1 for nowhere
    struct {
        float2 H[(MSMAX + 1) * MSMAX];  // column-major, leading dimension MSMAX + 1 (unrotated)
        float rc[MSMAX];                // rotations
        float2 rs[MSMAX], g[MSMAX + 1], d[MSMAX];
    } st;
    double tol2;  // square of the tolerance on ||r||
    float sc, beta;
    int ctl[4];
    unsigned long long mb[4];  // inbox 0, inbox 1, staged rows; [3]: the probe's, which nothing completes
    int fault;
    int fin[2][MAX_CLUSTER];   // faults of every CTA as published at a round's start (by its parity)
    int src[MAX_SITES][5];     // staged slot that holds the neighbour of each own site
    int hslot[MAX_SITES][4];   // slot of a neighbour owned by another CTA, -1 for an own site
    int nremote;
    int hsite[MAX_SITES * 4];  // GRID: site of each neighbour slot
    float anyf;                // GRID: faults of the projection exchange
#ifdef CP_PHASE_CLOCKS
    int acc_t[16];
#endif
};

__device__ __forceinline__ void st_async4(unsigned dst, unsigned x, unsigned y, unsigned z, unsigned w, unsigned bar) {
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];\n" ::"r"(dst),
        "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void mma16816(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                         unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// d = a b + c on two FP32 values at once
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n .reg .b64 a, b, c, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n mov.b64 c, {%6, %7};\n"
        " fma.rn.f32x2 d, a, b, c;\n mov.b64 {%0, %1}, d;\n}\n"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

__device__ __forceinline__ float4 both_orders(float2 v) { return make_float4(v.x, v.y, v.y, v.x); }

// GRID: a tagged pair of words, and a polled read of N of them (those with bit i of
// `have` clear are not read); false when the wait gave up
__device__ __forceinline__ void st_tagged(ulonglong2* p, unsigned x, unsigned y, unsigned tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};\n" ::"l"(p), "l"(t | x), "l"(t | y) : "memory");
}
__device__ __forceinline__ ulonglong2 ld_tagged(const ulonglong2* p) {
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];\n" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ bool tagged(const ulonglong2& v, unsigned tag) {
    return (unsigned)(v.x >> 32) == tag && (unsigned)(v.y >> 32) == tag;
}

// GRID: S.red / nrm as tc_reduce, from the CTAs' tagged partials gp[i][cta], i <= nd (and
// the fault sum of product nd + 1 into *anyf where that is not null); false when a wait
// gave up.  A warp takes values w and w + NW, all their partials (at most 160 CTAs) in
// flight at once.
constexpr int GRID_MAX = 160;
template <int NW>
__device__ __forceinline__ bool tc_reduce_grid(const ulonglong2* gp, int ncta, int nd, unsigned tag, long spin,
                                               float4* red, float* nrm, float* anyf) {
    constexpr int GP = GRID_MAX / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int last = nd + (anyf ? 1 : 0), n4 = max((nd + 4) & ~3, last + 1);
    bool ok = true;
#pragma unroll 1
    for (int i0 = warp; i0 < n4; i0 += 2 * NW) {
        ulonglong2 q[2][GP];
        unsigned wait = 0;  // bit h * GP + u: partial u of value i0 + h NW is still to come
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int u = 0; u < GP; ++u) {
                q[h][u] = make_ulonglong2(0, 0);
                if (i0 + h * NW <= last && lane + 32 * u < ncta) wait |= 1u << (h * GP + u);
            }
        for (long it = 0; wait && it < spin; ++it) {
#pragma unroll
            for (int b = 0; b < 2 * GP; ++b)
                if ((wait >> b) & 1u) q[b / GP][b % GP] = ld_tagged(gp + (long)(i0 + b / GP * NW) * ncta + lane + 32 * (b % GP));
#pragma unroll
            for (int b = 0; b < 2 * GP; ++b)
                if (((wait >> b) & 1u) && tagged(q[b / GP][b % GP], tag)) wait &= ~(1u << b);
        }
        ok = ok && wait == 0;
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = i0 + h * NW;
            float2 v = make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < GP; ++u) {
                v.x += __uint_as_float((unsigned)q[h][u].x);
                v.y += __uint_as_float((unsigned)q[h][u].y);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
                v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
            }
            if (lane == 0 && i < n4) {
                if (i == nd) *nrm = v.x;
                if (anyf && i == nd + 1) *anyf = v.x;
                red[i] = i < nd ? both_orders(v) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    }
    return ok;
}

// Partial inner products conj(X[i]) . y, i < nd, and |y|^2 as product nd, over the
// CTA's rows: a warp forms products 2w and 2w + 1 in one pass over y, two rows per
// 16-byte load, and sends both in one 16-byte st.async to every CTA's inbox (row =
// this CTA).  Packed FMAs: (Re Re, Im Im) and (Re Im, Im Re) of x and y are summed
// as they lie; Re and Im of the product are their sum and difference.
template <int NW, bool GRID>
__device__ __forceinline__ void tc_gram(const float2* X, long ldx, int nd, const float2* y, int npairs, unsigned inbox,
                                        int pw, unsigned bar, int nr, int me, ulonglong2* gp, unsigned tag) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float4* y4 = reinterpret_cast<const float4*>(y);
#pragma unroll 1
    for (int i0 = 2 * warp; i0 <= nd; i0 += 2 * NW) {
        // an odd count's partner repeats the norm
        const float4* xa = reinterpret_cast<const float4*>(i0 < nd ? X + (long)i0 * ldx : y);
        const float4* xb = reinterpret_cast<const float4*>(i0 + 1 < nd ? X + (long)(i0 + 1) * ldx : y);
        float2 ra = make_float2(0.f, 0.f), ia = ra, rb = ra, ib = ra;
#pragma unroll 3
        for (int e = lane; e < npairs; e += 32) {
            const float4 yv = y4[e], a = xa[e], b = xb[e];
            const float2 y0 = make_float2(yv.x, yv.y), y1 = make_float2(yv.z, yv.w);
            const float2 s0 = make_float2(yv.y, yv.x), s1 = make_float2(yv.w, yv.z);
            const float2 a0 = make_float2(a.x, a.y), a1 = make_float2(a.z, a.w);
            const float2 b0 = make_float2(b.x, b.y), b1 = make_float2(b.z, b.w);
            ra = fma2(a0, y0, ra);
            ia = fma2(a0, s0, ia);
            rb = fma2(b0, y0, rb);
            ib = fma2(b0, s0, ib);
            ra = fma2(a1, y1, ra);
            ia = fma2(a1, s1, ia);
            rb = fma2(b1, y1, rb);
            ib = fma2(b1, s1, ib);
        }
        const float2 pa = make_float2(ra.x + ra.y, ia.x - ia.y), pb = make_float2(rb.x + rb.y, ib.x - ib.y);
        // the lower half warp sums product i0, the upper one product i0 + 1
        const bool hi = lane & 16;
        float2 v = hi ? pb : pa;
        v.x += __shfl_xor_sync(0xffffffffu, hi ? pa.x : pb.x, 16);
        v.y += __shfl_xor_sync(0xffffffffu, hi ? pa.y : pb.y, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
            v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
        }
        if constexpr (GRID) {
            const int i = i0 + (lane >> 4);
            if ((lane & 15) == 0 && i <= nd)
                st_tagged(gp + (long)i * nr + me, __float_as_uint(v.x), __float_as_uint(v.y), tag);
            continue;
        }
        const float ox = __shfl_xor_sync(0xffffffffu, v.x, 16), oy = __shfl_xor_sync(0xffffffffu, v.y, 16);
        if (lane < nr)
            st_async4(cluster_addr(inbox + (unsigned)(me * pw + i0) * 8u, lane), __float_as_uint(v.x),
                      __float_as_uint(v.y), __float_as_uint(ox), __float_as_uint(oy), cluster_addr(bar, lane));
    }
}

// red[i] = sum over the inbox rows of column i, i < nd (and column nd into *nrm), half
// a warp a column, in one fixed tree (at most 16 rows): every CTA gets the same bits.
// red is zero from nd to the next multiple of four.
template <int NW>
__device__ __forceinline__ void tc_reduce(const float2* inbox, int rows, int pw, int nd, float4* red, float* nrm) {
    const int half = threadIdx.x >> 4, l = threadIdx.x & 15, n4 = (nd + 4) & ~3;
#pragma unroll 1
    for (int i = half; (i & ~1) < n4; i += 2 * NW) {
        float2 v = (l < rows && i <= nd) ? inbox[l * pw + i] : make_float2(0.f, 0.f);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
            v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
        }
        if (l == 0 && i < n4) {
            if (i == nd) *nrm = v.x;
            red[i] = i < nd ? both_orders(v) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}

// sum_{i < cnt} X[i ldx] coef[i], four rows at a time: coef is zero from cnt to the next
// multiple of four and the rows there are finite.  CLAMP: rows past the last are
// replaced by it.  Packed FMAs as in tc_gram.
template <bool CLAMP>
__device__ __forceinline__ float2 tc_combine(const float2* X, long ldx, const float4* coef, int cnt) {
    float2 p = make_float2(0.f, 0.f), q = p;
#pragma unroll 2
    for (int i = 0; i < cnt; i += 4) {
        float2 v[4];
        float4 h[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = X[(CLAMP ? (long)min(i + u, cnt - 1) : (long)u) * ldx];
#pragma unroll
        for (int u = 0; u < 4; ++u) h[u] = coef[i + u];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            p = fma2(v[u], make_float2(h[u].x, h[u].y), p);  // (Re Re, Im Im)
            q = fma2(v[u], make_float2(h[u].z, h[u].w), q);  // (Re Im, Im Re)
        }
        if (!CLAMP) X += 4 * ldx;
    }
    return make_float2(p.x - p.y, q.x + q.y);
}

#ifdef CP_PHASE_CLOCKS
__device__ unsigned tc_clock_launches = 0;
#define TC_STAMP(k)                          \
    do {                                     \
        if (clk) {                           \
            const long long now = clock64(); \
            S.acc_t[k] += (int)(now - t_prev); \
            t_prev = now;                    \
        }                                    \
    } while (0)
#else
#define TC_STAMP(k) \
    do {            \
    } while (0)
#endif

// NW warps.  NW = 8 serves at most 8 sites a CTA at two CTAs per SM, NW = 16 at most
// 16 (128 registers a thread either way).  PROBE: the test probe's wait comes first.  It is
// an instantiation of its own because its code, though never run, changed the others': a
// 384^2 solve 135.8 instead of 133.5 ms, 512^2 158.7 instead of 155.0, 256^2 51.9 instead of 51.8.
template <int NW, bool GRID, bool PROBE>
__global__ void __launch_bounds__(NW * 32, NW == 8 ? 2 : 1) k_coarse_tc(const __grid_constant__ CoopArgs<float> a,
                                                                        const __grid_constant__ TcShape g) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TcSmem& S = *reinterpret_cast<TcSmem*>(smem_raw);
    auto& st = S.st;
    float2* const inbox0 = reinterpret_cast<float2*>(smem_raw + g.o_inbox);
    unsigned* const Xs = reinterpret_cast<unsigned*>(smem_raw + g.o_x);
    float2* const V = reinterpret_cast<float2*>(smem_raw + g.o_v);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NT = NW * 32;
    // (a cluster launch has one cluster, so a CTA's rank in it is its block index)
    const int me = (int)blockIdx.x, ncta = (int)gridDim.x;
    const int nsite = a.Nx * a.Nt;
    const int s0 = me * g.spc;
    const int my_sites = max(0, min(nsite, s0 + g.spc) - s0);
    const int nrows = my_sites * NDOF;
    const int ldv = g.spc * NDOF;
    const int k = a.k, ms = a.ms;
    const int LD = MSMAX + 1;

    const unsigned base = GRID ? __ldcg(g.epoch) : 0u;
    unsigned ex = 0u, sx = 0u;  // GRID: exchanges and staged rows so far
    unsigned phases = 0u;  // parity of the next phase of barriers 0, 1, 2 (bits)
    // A wait that gives up marks the CTA faulted.  From then on the CTA skips its waits
    // and stops arming its barriers, and at the next round's cluster barrier every CTA
    // sees the fault and leaves the solve loop.
    // Only the last warp polls, the others wait at the CTA barrier that follows: polling
    // warps share the pipes of the shared-memory loads and shuffles of those still at work.
    auto flow_wait = [&](int b) {
        if (GRID || warp != NW - 1) return;
        const unsigned par = (phases >> b) & 1u;
        phases ^= 1u << b;
        if (mbar_wait(&S.mb[b], par, 1)) return;
        if (!S.fault && !mbar_wait(&S.mb[b], par, a.spin > 0 ? a.spin : FLOW_SPIN)) S.fault = 1;
    };
    auto arm = [&](int b, int bytes) {
        if (!GRID && tid == NT - 32 && !S.fault) mbar_arm(&S.mb[b], (unsigned)bytes);
    };

    // neighbour and push tables
    if (tid == 0) {
        if (!GRID) {
            for (int b = 0; b < 4; ++b) mbar_init(&S.mb[b], 1);
            asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        }
        S.fault = 0;
        int nrem = 0;
        for (int w = 0; w < my_sites; ++w) {
            S.src[w][0] = w;
            for (int d = 1; d < 5; ++d) {
                const int u = (int)nbr_site(s0 + w, d, a.Nx, a.Nt);
                const bool own = u / g.spc == me;
                S.hslot[w][d - 1] = own ? -1 : g.spc + nrem;
                S.src[w][d] = own ? u - s0 : g.spc + nrem;
                if (!own) S.hsite[nrem] = u;
                nrem += own ? 0 : 1;
            }
        }
        S.nremote = nrem;
        S.iters = 0;
        S.ctl[0] = 0;
#ifdef CP_PHASE_CLOCKS
        for (int i = 0; i < 16; ++i) S.acc_t[i] = 0;
#endif
    }
    for (int e = tid; e < 2 * MAX_CLUSTER; e += NT) (&S.fin[0][0])[e] = 0;
    if (!GRID) {
        cluster_arrive();
        cluster_wait();
    } else if (tid < my_sites) {  // own sites that another CTA reads (neighbours are mutual)
        int out = -1;
        for (int d = 1; d < 5; ++d)
            if ((int)nbr_site(s0 + tid, d, a.Nx, a.Nt) / g.spc != me) out = 0;
        S.push[tid][0] = out;
    }
    if (!GRID && tid < my_sites * 4) {
        const int w = tid >> 2, q = (tid & 3) + 1;
        const int from[5] = {0, 2, 1, 4, 3};  // dst = nbr(u, from[q]) reads u in direction q
        const int dst = (int)nbr_site(s0 + w, from[q], a.Nx, a.Nt), owner = dst / g.spc;
        int code = -1;
        if (owner != me) {
            int slot;
            const unsigned ra = cluster_addr(smem_addr(&S.hslot[dst - owner * g.spc][q - 1]), owner);
            asm volatile("ld.shared::cluster.b32 %0, [%1];\n" : "=r"(slot) : "r"(ra) : "memory");
            code = (owner << 16) | slot;
        }
        S.push[w][q - 1] = code;
    }
    {
        float2* Mp = reinterpret_cast<float2*>(smem_raw + g.o_m);
        for (int e = tid; e < k * (k + 1); e += NT) Mp[e] = from_d2<float>(a.pm->M[e]);
        for (int e = tid; e < (k + 1) * (k + 1); e += NT) Mp[k * (k + 1) + e] = from_d2<float>(a.pm->N[e]);
    }

    // operator fragments of site `warp`: entry (row i, column l) of direction d is word
    // (d 24 + l) 24 + i; columns 8 kt + 2 t and + 1 of K tile kt belong to lane (gq, t)
    const int gq = lane >> 2, t4 = lane & 3;
    const bool site_warp = warp < my_sites;
    unsigned fa[(5 - SD) * 3][4], fb[(5 - SD1) * 3][2];
    {
        uint4* opa = reinterpret_cast<uint4*>(smem_raw + g.o_op) + warp * OPA + lane;
        uint2* opb = reinterpret_cast<uint2*>(smem_raw + g.o_op + g.spc * OPA * 16) + warp * OPB + lane;
        const unsigned* Ab = a.Ah + (long)(s0 + (site_warp ? warp : 0)) * (5 * NDOF * NDOF) + gq;
#pragma unroll
        for (int d = 0; d < 5; ++d)
#pragma unroll
            for (int kt = 0; kt < 3; ++kt) {
                const unsigned* p = Ab + (d * NDOF + 8 * kt + 2 * t4) * NDOF;
                const uint4 qa = make_uint4(__ldg(p), __ldg(p + 8), __ldg(p + NDOF), __ldg(p + NDOF + 8));
                const uint2 qb = make_uint2(__ldg(p + 16), __ldg(p + NDOF + 16));
                if (d < SD) {
                    if (site_warp) opa[(d * 3 + kt) * 32] = qa;
                } else {
                    unsigned* q = fa[(d - SD) * 3 + kt];
                    q[0] = qa.x, q[1] = qa.y, q[2] = qa.z, q[3] = qa.w;
                }
                if (d < SD1) {
                    if (site_warp) opb[(d * 3 + kt) * 32] = qb;
                } else {
                    unsigned* q = fb[(d - SD1) * 3 + kt];
                    q[0] = qb.x, q[1] = qb.y;
                }
            }
    }
    // the deflation space on the own rows
    if (g.ws) {
        float2* Ws = reinterpret_cast<float2*>(smem_raw + g.o_w);
        const float2* Wl = a.W + (long)s0 * NDOF;
        for (int i = 0; i <= k; ++i)
            for (int e = tid; e < nrows; e += NT) Ws[i * ldv + e] = Wl[(long)i * nsite * NDOF + e];
    }

    // thread tid owns row tid; row 0 of V holds r at a round's start
    const bool row_on = tid < nrows;
    float2* const xs = reinterpret_cast<float2*>(smem_raw + g.o_sol);
    for (int e = tid; e < g.vrows * ldv; e += NT) V[e] = make_float2(0.f, 0.f);
    __syncthreads();
    if (row_on) {
        xs[tid] = make_float2(0.f, 0.f);
        V[tid] = a.f[(long)s0 * NDOF + tid];
    }
    __syncthreads();
    if constexpr (PROBE) {  // test probe: a wait that nothing ends gives up
        const long spin = a.spin > 0 ? a.spin : FLOW_SPIN;
        if constexpr (GRID) {
            if (tid == 0) {
                long it = 0;
                while (it < spin && __ldcg(g.epoch + 1) == 0u) ++it;
                if (it == spin) S.fault = 1;
            }
        } else if (!S.fault && !mbar_wait(&S.mb[3], 0u, spin)) {
            S.fault = 1;
        }
        __syncthreads();
    }
    // a new basis row: an even row stages itself and its odd partner, in the own
    // site's slot and in those of the neighbouring CTAs that read it
    auto stage = [&](float2 v) {
        const __half2 h = __floats2half2_rn(v.x * TC_XS, v.y * TC_XS);
        const float2 hf = __half22float2(h);
        // v 2^10 - hi is exact in FP32 (hi is v 2^10 rounded to 11 bits)
        const __half2 l = __floats2half2_rn(fmaf(v.x, TC_XS, -hf.x) * TC_RS, fmaf(v.y, TC_XS, -hf.y) * TC_RS);
        const unsigned hi = *reinterpret_cast<const unsigned*>(&h), lo = *reinterpret_cast<const unsigned*>(&l);
        const unsigned hi1 = __shfl_down_sync(0xffffffffu, hi, 1), lo1 = __shfl_down_sync(0xffffffffu, lo, 1);
        if (row_on && !(lane & 1)) {
            const int site = tid / NDOF, off = (tid - site * NDOF) * 2;
            *reinterpret_cast<uint4*>(Xs + site * XW + off) = make_uint4(hi, hi1, lo, lo1);
            if constexpr (GRID) {
                if (S.push[site][0] >= 0) {
                    ulonglong2* dst = g.rows + ((long)(sx & 1u) * nsite + s0) * NDOF + tid;
                    st_tagged(dst, hi, lo, base + sx + 1u);
                    st_tagged(dst + 1, hi1, lo1, base + sx + 1u);
                }
                return;
            }
            const int4 p = *reinterpret_cast<const int4*>(S.push[site]);
            auto send = [&](int code) {
                if (code < 0) return;
                const int owner = code >> 16;
                st_async4(cluster_addr(smem_addr(Xs + (code & 0xffff) * XW + off), owner), hi, hi1, lo, lo1,
                          cluster_addr(smem_addr(&S.mb[2]), owner));
            };
            send(p.x);
            send(p.y);
            send(p.z);
            send(p.w);
        }
    };
#ifdef CP_PHASE_CLOCKS
    const bool clk = me == 0 && tid == 0 && atomicAdd(&tc_clock_launches, 1u) < 48u;
    long long t_prev = clock64();
    int clk_steps = 0;
#endif
    // one exchange of nd inner products of X with y into S.red[buf], and |y|^2.  The
    // buffers alternate: a CTA sends into buffer b only after an exchange on the other
    // one, to which this CTA contributes after it has read buffer b.
    auto exchange = [&](int buf, const float2* X, long ldx, int nd, const float2* y, bool faults = false) {
        arm(buf, ncta * ((nd + 2) & ~1) * 8);
        const unsigned in = smem_addr(inbox0) + (unsigned)(buf * MAX_CLUSTER * g.pw) * 8u;
        ulonglong2* gp = GRID ? g.part + (long)(ex & 1u) * PSTR * ncta : nullptr;
        tc_gram<NW, GRID>(X, ldx, nd, y, nrows >> 1, in, g.pw, smem_addr(&S.mb[buf]), ncta, me, gp, base + ex + 1u);
        TC_STAMP(8);
        if constexpr (GRID) {
            if (faults && tid == NT - 1)
                st_tagged(gp + (long)(nd + 1) * ncta + me, __float_as_uint(S.fault ? 1.f : 0.f), 0u, base + ex + 1u);
            const long spin = S.fault ? 0 : (a.spin > 0 ? a.spin : FLOW_SPIN);
            if (!tc_reduce_grid<NW>(gp, ncta, nd, base + ex + 1u, spin, S.red[buf], &S.nrm[buf],
                                    faults ? &S.anyf : nullptr))
                S.fault = 1;
            ++ex;
        } else {
            flow_wait(buf);
            __syncthreads();
            TC_STAMP(9);
            tc_reduce<NW>(inbox0 + buf * MAX_CLUSTER * g.pw, ncta, g.pw, nd, S.red[buf], &S.nrm[buf]);
        }
        __syncthreads();
    };
    // GRID: the neighbouring CTAs' rows of the staged vector into their slots
    auto receive = [&]() {
        if constexpr (GRID) {
            const ulonglong2* src = g.rows + (long)(sx & 1u) * nsite * NDOF;
            for (int e = tid; e < S.nremote * (NDOF / 2); e += NT) {
                const int slot = e / (NDOF / 2), m = e - slot * (NDOF / 2);
                const ulonglong2* p = src + (long)S.hsite[slot] * NDOF + 2 * m;
                ulonglong2 q0, q1;
                long it = S.fault ? 0 : (a.spin > 0 ? a.spin : FLOW_SPIN);
                do {
                    q0 = ld_tagged(p);
                    q1 = ld_tagged(p + 1);
                } while (!(tagged(q0, base + sx + 1u) && tagged(q1, base + sx + 1u)) && --it > 0);
                if (it <= 0) S.fault = 1;
                *reinterpret_cast<uint4*>(Xs + (g.spc + slot) * XW + m * 4) =
                    make_uint4((unsigned)q0.x, (unsigned)q1.x, (unsigned)q0.y, (unsigned)q1.y);
            }
            ++sx;
        }
    };
    int cycles = 0;
    // Least squares of the cycle, by the last warp while the staged rows travel.  The
    // rotations turn column j's running entry into p_{t+1} = c_t h_{t+1} - conj(s_t) p_t,
    // so the entry that meets h_{j+1,j} is a dot product p = sum_i u_i h_i with
    // u^{(j+1)} = (-conj(s_j) u^{(j)}, c_j): lane i has u_i, and a step costs one
    // warp sum instead of a chain of j rotations.  The rotated columns themselves are
    // formed at the cycle's end, one lane a column.
    auto ls_update = [&](int jc, float hnv) {
        float2 h = make_float2(0.f, 0.f);
        if (lane <= jc) {
            const float4 h0 = S.red[0][lane], h1 = S.red[1][lane];
            h = make_float2(h1.x + h0.x, h1.y + h0.y);
            st.H[lane + LD * jc] = h;
        } else if (lane == jc + 1) {
            st.H[lane + LD * jc] = make_float2(hnv, 0.f);
        }
        float2 u_ls = S.u_ls[lane], g_ls = S.g_ls;
        if (jc == 0) {
            u_ls = make_float2(lane == 0 ? 1.f : 0.f, 0.f);
            g_ls = make_float2(S.beta, 0.f);
        }
        float2 p = cmul(u_ls, h);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            p.x += __shfl_xor_sync(0xffffffffu, p.x, o);
            p.y += __shfl_xor_sync(0xffffffffu, p.y, o);
        }
        float cc;
        float2 ss, rv;
        givens_real_<float>(p, hnv, cc, ss, rv);
        const float2 ms_c = cneg(conj_(ss));
        S.u_ls[lane] = lane == jc + 1 ? make_float2(cc, 0.f) : cmul(ms_c, u_ls);
        const float2 gj = cscale(g_ls, cc);
        g_ls = cmul(ms_c, g_ls);
        __syncwarp();
        if (lane == 0) {
            S.g_ls = g_ls;
            st.rc[jc] = cc;
            st.rs[jc] = ss;
            st.g[jc] = gj;
            S.ctl[0] = ((double)(g_ls.x * g_ls.x + g_ls.y * g_ls.y) <= S.tol2) ? 1 : 0;
            S.ctl[1] = (hnv == 0.f) ? 1 : 0;
        }
    };

    while (true) {
        // ---- projection onto the deflation space: d = argmin ||W^+ r - H_k d|| ----
        // Every CTA publishes its fault to all before the split cluster barrier; all
        // read the same flags after it, the one place where CTAs leave.
        if (!GRID) {
            if (warp == 0 && lane < ncta) {
                const unsigned ra = cluster_addr(smem_addr(&S.fin[cycles & 1][me]), lane);
                asm volatile("st.shared::cluster.b32 [%0], %1;\n" ::"r"(ra), "r"(S.fault) : "memory");
            }
            __syncwarp();
            cluster_arrive();
        }
        const float2* Wl = g.ws ? reinterpret_cast<const float2*>(smem_raw + g.o_w) : a.W + (long)s0 * NDOF;
        const long ldw = g.ws ? ldv : (long)nsite * NDOF;
        exchange(0, Wl, ldw, k + 1, V, true);
        if (!GRID) cluster_wait();
        int anyf = 0;
        if (GRID) anyf = S.fault | (S.anyf != 0.f);
        else
            for (int q = 0; q < ncta; ++q) anyf |= S.fin[cycles & 1][q];
        // S.ctl[0]: the last cycle converged (the same in every CTA that has not faulted)
        if (anyf | S.ctl[0] | (cycles >= a.max_cycles)) break;
        if (cycles == 0 && tid == 0)  // r = f: the tolerance is relative to ||f||
            S.tol2 = a.tol * a.tol * (double)fmaxf(S.nrm[0], 0.f);
        {
            const float2* Mp = reinterpret_cast<const float2*>(smem_raw + g.o_m);
            const float2* Np = Mp + k * (k + 1);
#pragma unroll 1
            for (int i = warp; i <= k; i += NW) {  // pd = M g, pu = N g: warp i takes row i
                float2 pd = make_float2(0.f, 0.f), pu = pd;
                for (int l = lane; l <= k; l += 32) {
                    const float4 g4 = S.red[0][l];
                    const float2 gl = make_float2(g4.x, g4.y);
                    if (i < k) pd = cfma(Mp[i + k * l], gl, pd);
                    pu = cfma(Np[i + (k + 1) * l], gl, pu);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    pd.x += __shfl_xor_sync(0xffffffffu, pd.x, o);
                    pd.y += __shfl_xor_sync(0xffffffffu, pd.y, o);
                    pu.x += __shfl_xor_sync(0xffffffffu, pu.x, o);
                    pu.y += __shfl_xor_sync(0xffffffffu, pu.y, o);
                }
                if (lane == 0) {  // (row k of M is none: a zero coefficient)
                    S.coef[0][i] = both_orders(i < k ? pd : make_float2(0.f, 0.f));
                    S.coef[1][i] = both_orders(pu);
                }
            }
        }
        if (tid < 3) S.coef[0][k + 1 + tid] = S.coef[1][k + 1 + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        if (row_on) {
            xs[tid] = cadd(xs[tid], tc_combine<true>(Wl + tid, ldw, S.coef[0], k + 1));
            V[tid] = csub(V[tid], tc_combine<true>(Wl + tid, ldw, S.coef[1], k + 1));
        }
        __syncthreads();
        exchange(1, V, ldv, 0, V);
        // beta = ||r||, the stop test (on squares), and the start of the cycle; the scale, an
        // FP64 reciprocal root rounded to FP32, on another warp
        const float b2 = fmaxf(S.nrm[1], 0.f);
        if (tid == 0) {
            S.ctl[0] = ((double)b2 <= S.tol2 || b2 == 0.f) ? 1 : 0;
            S.ctl[1] = 0;
            S.beta = sqrtf(b2);
        }
        if (tid == 32) S.sc = b2 > 0.f ? (float)rsqrt((double)b2) : 0.f;
        __syncthreads();
        if (S.ctl[0]) continue;  // converged: leave at the next round's barrier
        // ---- one GMRES(ms) cycle from r ----
        arm(2, S.nremote * XW * 4);
        {
            float2 v = make_float2(0.f, 0.f);
            if (row_on) V[tid] = v = cscale(V[tid], S.sc);
            stage(v);
        }
        int j = 0;
        TC_STAMP(7);
#pragma unroll 1
        for (; j < ms; ++j) {
            float2* const wl = V + (j + 1) * ldv;
            flow_wait(2);     // v_j staged by the neighbouring CTAs
            receive();
            __syncthreads();  // and by the own warps
            TC_STAMP(0);
            if (site_warp) {  // w = A v_j at site `warp`
                float c0[2][4], c1[2][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) c0[0][u] = c0[1][u] = c1[0][u] = c1[1][u] = 0.f;
                const uint4* opa = reinterpret_cast<const uint4*>(smem_raw + g.o_op) + warp * OPA + lane;
                const uint2* opb =
                    reinterpret_cast<const uint2*>(smem_raw + g.o_op + g.spc * OPA * 16) + warp * OPB + lane;
                // column n = gq & 3 of the real form: n = 0: (Re, -Im) of hi, 1: (Im, Re) of hi,
                // 2 and 3: the same of lo (columns 4..7 repeat them)
                const unsigned sel = (gq & 1) ? 0x1032u : 0x3210u, sgn = (gq & 1) ? 0u : 0x80000000u;
                const unsigned* xl = Xs + t4 * 4 + (gq & 2);
#pragma unroll
                for (int d = 0; d < 5; ++d) {
                    const unsigned* xp = xl + S.src[warp][d] * XW;
#pragma unroll
                    for (int kt = 0; kt < 3; ++kt) {
                        const uint2 x = *reinterpret_cast<const uint2*>(xp + kt * 16);
                        const unsigned b0 = __byte_perm(x.x, 0u, sel) ^ sgn, b1 = __byte_perm(x.y, 0u, sel) ^ sgn;
                        const int u = (d * 3 + kt) & 1;
                        uint4 qa;
                        uint2 qb;
                        if (d < SD) {
                            qa = opa[(d * 3 + kt) * 32];
                        } else {
                            const unsigned* q = fa[(d - SD) * 3 + kt];
                            qa = make_uint4(q[0], q[1], q[2], q[3]);
                        }
                        if (d < SD1) {
                            qb = opb[(d * 3 + kt) * 32];
                        } else {
                            const unsigned* q = fb[(d - SD1) * 3 + kt];
                            qb = make_uint2(q[0], q[1]);
                        }
                        mma16816(c0[u], qa.x, qa.y, qa.z, qa.w, b0, b1);
                        mma16816(c1[u], qb.x, 0u, qb.y, 0u, b0, b1);
                    }
                }
                // lane t = 0 holds columns 0, 1 (hi) and t = 1 columns 2, 3 (lo) of rows gq,
                // gq + 8 (c0) and 16 + gq (c1); lanes t = 2, 3 repeat them
                float o[6] = {c0[0][0] + c0[1][0], c0[0][1] + c0[1][1], c0[0][2] + c0[1][2],
                              c0[0][3] + c0[1][3], c1[0][0] + c1[1][0], c1[0][1] + c1[1][1]};
#pragma unroll
                for (int u = 0; u < 6; ++u) {
                    o[u] *= (t4 & 1) ? TC_XRS_INV : TC_XS_INV;
                    o[u] += __shfl_xor_sync(0xffffffffu, o[u], 1);
                }
                // lane t writes row gq + 8 t (t < 3)
                if (t4 < 3)
                    wl[warp * NDOF + gq + 8 * t4] =
                        make_float2(t4 == 0 ? o[0] : t4 == 1 ? o[2] : o[4], t4 == 0 ? o[1] : t4 == 1 ? o[3] : o[5]);
            }
            __syncthreads();
            TC_STAMP(1);
            // step j - 1's least-squares update is complete; a stop discards step j: j columns
            if (j > 0 && (S.ctl[0] | S.ctl[1])) break;
            // CGS2: two passes of h = V^+ w, w -= V h
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {
                exchange(pass, V, ldv, j + 1, wl);
                TC_STAMP(2);
                if (pass == 0) {
                    if (row_on) wl[tid] = csub(wl[tid], tc_combine<false>(V + tid, ldv, S.red[0], j + 1));
                    __syncthreads();
                    TC_STAMP(3);
                }
            }
            // h_{j+1,j} = ||w - V h2|| = sqrt(n2 - |h2|^2) (V orthonormal), the same bits in
            // every thread; then v_{j+1} = (w - V h2) / h_{j+1,j}.
            float h2n = 0.f;
            if (lane <= j) {
                const float4 h = S.red[1][lane];
                h2n = h.x * h.x + h.y * h.y;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) h2n += __shfl_xor_sync(0xffffffffu, h2n, o);
            const float hh = fmaxf(S.nrm[1] - h2n, 0.f);
            TC_STAMP(10);
            arm(2, S.nremote * XW * 4);
            if (warp * 32 < nrows) {
                float2 v = make_float2(0.f, 0.f);
                if (row_on) {
                    // the rows need the reciprocal root and the least squares (a warp without rows)
                    // the root: each forms its own
                    const float inv = hh > 0.f ? __frsqrt_rn(hh) : 0.f;
                    v = cscale(csub(wl[tid], tc_combine<false>(V + tid, ldv, S.red[1], j + 1)), inv);
                    wl[tid] = v;
                }
                TC_STAMP(11);
                stage(v);
            }
            if (warp == NW - 1) ls_update(j, sqrtf(hh));
            TC_STAMP(5);
#ifdef CP_PHASE_CLOCKS
            ++clk_steps;
#endif
        }
        if (j == ms) {     // the last step's update, when no stop came before
            flow_wait(2);  // the staging of v_ms, which no apply reads
            ++sx;
            __syncthreads();
        }
        if (tid == 0) S.iters += j;
        TC_STAMP(12);
        // ---- finish the cycle: d = R^{-1} g, rho = c - H d, x += V d, r = V rho ----
        if (warp == 0) {
            // R is formed over the staged slots, which nothing reads or sends to before the
            // next cycle's norm exchange
            float2* Rm = reinterpret_cast<float2*>(Xs);
            if (lane < j) {  // column `lane` of R: the rotations applied to that column of H
                const float2* Hc = st.H + LD * lane;
                float2 p = Hc[0];
                for (int t = 0; t <= lane; ++t) {
                    float2 q = Hc[t + 1];
                    rot_<float>(st.rc[t], st.rs[t], p, q);
                    Rm[t + LD * lane] = p;
                    p = q;
                }
            }
            __syncwarp();
            back_subst_warp<float>(Rm, st.g, st.d, j, lane);
            __syncwarp();
            float2 acc = make_float2(lane == 0 ? S.beta : 0.f, 0.f);
            if (lane <= j)  // H is zero below its subdiagonal
                for (int l = max(lane - 1, 0); l < j; ++l) acc = cfms_<float>(st.H[lane + LD * l], st.d[l], acc);
            S.coef[0][lane] = both_orders(lane < j ? st.d[lane] : make_float2(0.f, 0.f));
            S.coef[1][lane] = both_orders(lane <= j ? acc : make_float2(0.f, 0.f));
        }
        __syncthreads();
        TC_STAMP(13);
        if (row_on) {
            xs[tid] = cadd(xs[tid], tc_combine<false>(V + tid, ldv, S.coef[0], j));
            V[tid] = tc_combine<true>(V + tid, ldv, S.coef[1], j + 1);
        }
        ++cycles;
        __syncthreads();  // (a stop is taken after the next exchange)
        TC_STAMP(6);
    }
    if (row_on) a.x[(long)s0 * NDOF + tid] = xs[tid];
    __syncthreads();
    if (tid == 0 && S.fault) atomicAdd(reinterpret_cast<unsigned long long*>(&a.out->timeouts), 1ULL);
    if (me == 0 && tid == 0) {
        a.out->iters += S.iters;
        a.out->cycles += cycles;
        a.out->solves += 1;
        a.out->unconverged += S.ctl[0] ? 0 : 1;
        a.out->ctas = ncta;
        a.out->spc = g.spc;
        a.out->flow = 1;
        a.out->dc = 0;
        a.out->ash = 1;
        a.out->half = 1;
        a.out->paired = 0;
        a.out->mma = 1;
    }
#ifdef CP_PHASE_CLOCKS
    if (clk && clk_steps > 0)
        printf("coarse_tc phases (cycles/step over %d steps): staging wait %d, apply %d, gram %d, exchange wait %d, "
               "reduce %d, update %d, norm %d, v %d, stage %d, cycle end %d + %d + %d, cycle start %d\n",
               clk_steps, S.acc_t[0] / clk_steps, S.acc_t[1] / clk_steps, S.acc_t[8] / clk_steps, S.acc_t[9] / clk_steps,
               S.acc_t[2] / clk_steps, S.acc_t[3] / clk_steps, S.acc_t[10] / clk_steps, S.acc_t[11] / clk_steps,
               S.acc_t[5] / clk_steps, S.acc_t[12] / clk_steps, S.acc_t[13] / clk_steps, S.acc_t[6] / clk_steps,
               S.acc_t[7] / clk_steps);
#endif
    if (GRID) {
        // (every CTA has read the base: this one has had a whole exchange from all of them)
        if (me == 0 && tid == 0) *g.epoch = base + max(ex, sx) + 1u;
    } else {
        cluster_arrive();  // no CTA leaves while others may still write its shared memory
        cluster_wait();
    }
}

struct TcGeometry {
    int ok = 0, ctas = 0, nw = 0, grid = 0, at_once = 1;
    size_t smem = 0;
    TcShape g{};
};

// remote neighbours of the CTA with the most of them
int max_halo(int Nx, int Nt, int spc) {
    const int nsite = Nx * Nt;
    int most = 0;
    for (int s0 = 0; s0 < nsite; s0 += spc) {
        int c = 0;
        for (int s = s0; s < std::min(nsite, s0 + spc); ++s)
            for (int d = 1; d < 5; ++d) {
                const int xx = s % Nx, t = s / Nx;
                const int u = d == 1 ? (xx + 1 == Nx ? s - xx : s + 1)
                            : d == 2 ? (xx == 0 ? s + Nx - 1 : s - 1)
                            : d == 3 ? (t + 1 == Nt ? xx : s + Nx)
                                     : (t == 0 ? s + Nx * (Nt - 1) : s - Nx);
                if (u < s0 || u >= s0 + spc) ++c;
            }
        most = std::max(most, c);
    }
    return most;
}

// the shared memory and, of the cluster form, the cluster size that a kernel may have
template <int NW, bool GRID, bool PROBE>
bool allow() {
    auto* kern = k_coarse_tc<NW, GRID, PROBE>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_LIMIT) == cudaSuccess &&
        (GRID || cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess))
        return true;
    (void)cudaGetLastError();
    return false;
}

template <int NW>
bool fits(TcGeometry& G) {
    auto* kern = k_coarse_tc<NW, false, false>;
    if (!allow<NW, false, false>()) return false;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = G.ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(G.ctas);
    cfg.blockDim = dim3(NW * 32);
    cfg.dynamicSmemBytes = G.smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, kern, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return nc >= 1;
}

// shared-memory layout for spc sites a CTA; two: leave room for two CTAs per SM when
// that costs only the deflation space's copy
void tc_layout(int Nx, int Nt, int ms, int k, int spc, bool two, TcGeometry& G) {
    TcShape& g = G.g;
    g = TcShape{};
    g.spc = spc;
    G.ctas = (Nx * Nt + spc - 1) / spc;
    // an inbox row holds its products and the norm, in 16-byte pairs; rows an odd
    // number of pairs apart fall on different banks
    g.pw = (std::max(k + 2, ms + 1) + 1) & ~1;
    if (g.pw % 4 == 0) g.pw += 2;
    g.halo = max_halo(Nx, Nt, spc);
    size_t o = (sizeof(TcSmem) + 15) & ~size_t(15);
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = (o + bytes + 15) & ~size_t(15);
        return (int)at;
    };
    const size_t rows = (size_t)spc * NDOF;
    g.o_inbox = take(G.grid ? 0 : (size_t)2 * MAX_CLUSTER * g.pw * sizeof(float2));
    g.o_x = take(std::max((size_t)(spc + g.halo) * XW * 4, (size_t)(MSMAX + 1) * MSMAX * sizeof(float2)));
    g.vrows = std::max(ms + 1, (ms + 3) & ~3);  // row updates read whole groups of four rows
    g.o_v = take((size_t)g.vrows * rows * sizeof(float2));
    g.o_sol = take(rows * sizeof(float2));
    g.o_m = take((size_t)(2 * k + 1) * (k + 1) * sizeof(float2));
    g.o_op = take((size_t)spc * (OPA * 16 + OPB * 8));
    const size_t base = o, with_w = o + (size_t)(k + 1) * rows * sizeof(float2);
    const size_t half = (SMEM_LIMIT - 1024) / 2;
    g.ws = (with_w <= half || (with_w <= SMEM_LIMIT && (!two || base > half))) ? 1 : 0;
    g.o_w = (int)base;
    G.smem = g.ws ? with_w : base;
}

constexpr int GRID_SPC = 8;  // grid form: sites a CTA, at least
// A step of the grid form, and of coarse_coop.cu's cluster kernel by its sites (18.1 us at
// 24^2, 29.9 us at 32^2); that kernel's 16-CTA clusters that are resident at once
constexpr long GRID_STEP_NS = 14000, CLUSTER_STEP_NS = 2900, CLUSTER_SITE_NS = 26;
constexpr int CLUSTERS = 7;

void tc_geometry_uncached(int Nx, int Nt, int ms, int k, int peers, TcGeometry& G) {
    const int nsite = Nx * Nt;
    if (nsite <= MAX_CLUSTER * MAX_SITES) {
        for (int cl = MAX_CLUSTER; cl >= 1; cl >>= 1) {
            const int spc = (nsite + cl - 1) / cl;
            if (spc > MAX_SITES) return;
            G.nw = spc <= 8 ? 8 : 16;
            tc_layout(Nx, Nt, ms, k, spc, G.nw == 8, G);
            if (G.smem > SMEM_LIMIT) continue;
            G.ok = (G.nw == 8 ? fits<8>(G) : fits<16>(G)) ? 1 : 0;
            if (G.ok) return;
        }
        return;
    }
    // Grid form.  A step takes about as long with eight sites a CTA as with 16 (384^2: 13.3
    // and 14 us), but a solve then holds twice the SMs, and of solves that run at once only as
    // many go on as fit: eight sites where all peers' grids fit beside one another, else 16.
    // Where not even those fit, the cluster kernel (16 CTAs; its step grows with the grid) may
    // serve the peers sooner: the form with the smaller time a step over the number at once.
    // Mixed solves, ms each, 8 | 16 sites a CTA | cluster kernel: 7 at once, 320^2 45 | 26 | 25,
    // 384^2 68 | 39 | 32, 512^2 156 | 79 | 58; 3 at once, 48 | 46 | 50, 69 | 52 | 64,
    // 152 | 77 | 112; alone, 130 | 127 | 141, 137 | 141 | 179, 157 | 159 | 319.
    const int sms = sm_count(), most = std::min(sms, GRID_MAX);
    const int least = (nsite + most - 1) / most;
    if (least > MAX_SITES) return;
    if (!allow<16, true, false>()) return;
    for (int spc : {std::max(GRID_SPC, least), MAX_SITES}) {
        TcGeometry C;
        C.nw = 16;
        C.grid = 1;
        tc_layout(Nx, Nt, ms, k, spc, false, C);
        if (C.smem > SMEM_LIMIT) continue;
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_coarse_tc<16, true, false>, 512, C.smem) !=
            cudaSuccess) {
            (void)cudaGetLastError();
            return;
        }
        const int at_once = per_sm * sms / C.ctas;
        if (at_once < 1) continue;
        C.ok = 1;
        C.at_once = at_once;
        G = C;
        if (at_once >= peers) return;
    }
    if (!G.ok) return;
    const long grids = std::min(peers, G.at_once), clusters = std::min(peers, CLUSTERS);
    if (GRID_STEP_NS * clusters > (CLUSTER_STEP_NS + CLUSTER_SITE_NS * nsite) * grids) G.ok = 0;
}

}  // namespace

mg_status launch_coarse_tc(const CoopArgs<float>& a, cudaStream_t s, bool* launched) {
    *launched = false;
    if (!a.Ah || !a.mma || a.dc || (long)a.Nx * a.Nt > (long)GRID_MAX * MAX_SITES) return MG_OK;
    struct Entry {
        int dev, Nx, Nt, ms, k, peers;
        TcGeometry G;
    };
    static std::mutex mu;
    static std::vector<Entry> cache;
    // (within one cluster's sites the peers change nothing)
    const int peers = a.Nx * a.Nt > MAX_CLUSTER * MAX_SITES ? std::min(std::max(a.peers, 1), GRID_MAX) : 1;
    int dev = 0;
    MG_CUDA_TRY(cudaGetDevice(&dev));
    TcGeometry G;
    {
        std::lock_guard<std::mutex> lock(mu);
        bool hit = false;
        for (const Entry& e : cache)
            if (e.dev == dev && e.Nx == a.Nx && e.Nt == a.Nt && e.ms == a.ms && e.k == a.k &&
                e.peers == peers) {
                G = e.G;
                hit = true;
                break;
            }
        if (!hit) {
            tc_geometry_uncached(a.Nx, a.Nt, a.ms, a.k, peers, G);
            cache.push_back(Entry{dev, a.Nx, a.Nt, a.ms, a.k, peers, G});
        }
    }
    if (!G.ok || (G.grid && (!a.part || !a.rows || G.ctas > a.part_ctas))) return MG_OK;
    G.g.part = reinterpret_cast<ulonglong2*>(a.part);
    G.g.rows = reinterpret_cast<ulonglong2*>(a.rows);
    G.g.epoch = a.epoch;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    if (G.grid) {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    } else {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = G.ctas;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    }
    cfg.gridDim = dim3(G.ctas);
    cfg.blockDim = dim3(G.nw * 32);
    cfg.dynamicSmemBytes = G.smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (a.probe) {
        const bool ok = G.grid ? allow<16, true, true>() : G.nw == 8 ? allow<8, false, true>() : allow<16, false, true>();
        if (!ok) return set_error("coarse solve: the probed kernel cannot run here"), MG_ECUDA;
        if (G.grid) MG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_coarse_tc<16, true, true>, a, G.g));
        else if (G.nw == 8) MG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_coarse_tc<8, false, true>, a, G.g));
        else MG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_coarse_tc<16, false, true>, a, G.g));
    } else if (G.grid) {
        MG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_coarse_tc<16, true, false>, a, G.g));
    } else if (G.nw == 8) {
        MG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_coarse_tc<8, false, false>, a, G.g));
    } else {
        MG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_coarse_tc<16, false, false>, a, G.g));
    }
    count_launch();
    *launched = true;
    return MG_OK;
}

}  // namespace mg
