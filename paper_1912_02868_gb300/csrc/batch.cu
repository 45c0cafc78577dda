// Kernels of the lockstep multi-right-hand-side solve (batch.cuh):
//  * batched inner products, multi-vector updates, norms and scalings, one
//    launch for a whole block of right-hand sides, each right-hand side reduced
//    deterministically (fixed per-thread order, fixed shuffle tree, the chunk
//    partials added in chunk order by the last chunk of that right-hand side);
//  * the 24-dof block stencil of the intermediate and coarsest grids
//    (D^ = P^+ D P, Section 2) for a block of right-hand sides on tensor cores.
//
// Tensor-core block products.  For one site s and one direction d the 5-point
// stencil multiplies a complex 24 x 24 block A by the complex 24-vectors of
// eight right-hand sides at the neighbour: a complex (24 x 24)(24 x 8) product.
// With the real embedding that keeps real and imaginary parts interleaved,
//   [re y_a]   [re A_ac  -im A_ac] [re x_c]
//   [im y_a] = [im A_ac   re A_ac] [im x_c],
// the product is a real (48 x 48)(48 x 8) one, i.e. 3 x 3 tiles of
// mma.sync.m16n8k16 (BF16 or FP16 inputs, FP32 accumulation), and the vector's
// natural layout (re, im, re, im, ...) is exactly the K order of the B operand.
// The operator is stored once per apply-format as complex 16-bit pairs in the
// order the A fragments are loaded (one 8-byte load per thread per tile): a
// thread's rows g and g + 8 of a real tile are the two forms of one complex row,
// so both come from the same words by a sign flip and a half swap in registers.  The FP32
// vectors are split into x = hi + lo, both rounded to the 16-bit format, and
// multiplied twice, so the product carries the operator's rounding only.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <atomic>
#include <type_traits>

#include "batch.cuh"

namespace mg {

namespace {

// ------------------------------------------------------------ batched BLAS --

template <typename T>
__device__ __forceinline__ C2<T> bblock_sum(C2<T> v, C2<T>* sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    __syncthreads();
    if (lane == 0) sm[warp] = v;
    __syncthreads();
    C2<T> r = mk<T>(0, 0);
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r = cadd(r, sm[w]);
    return r;
}

// Sums over the block of CH complex values a thread holds in acc: value c is returned
// (valid in threads 2c: real part, 2c + 1: imaginary part, in *out).  A warp's butterfly
// halves the values it carries at each stage (2 CH - 1 + log2(32 / 2 CH) additions a
// lane instead of 10 CH), which matters most in FP64, where an addition of a warp holds
// its scheduler for 64 cycles; the warps' sums are added in warp order.  k_bgram took
// 66 ms of a 256^2 solve of 64 right-hand sides, 45 ms so (FP64, 131072 entries x 64:
// 396 us a launch; FP32: 27 us).
template <typename T, int CH>
__device__ __forceinline__ T bblock_sums(const C2<T> (&acc)[CH], T (*sm)[2 * CH]) {
    constexpr int NVAL = 2 * CH;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T v[NVAL];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        v[2 * c] = acc[c].x;
        v[2 * c + 1] = acc[c].y;
    }
    int idx = 0;  // the value this lane ends with
#pragma unroll
    for (int half = NVAL / 2, o = 16; half > 0; half >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const T send = up ? v[i] : v[i + half];
            v[i] = (up ? v[i + half] : v[i]) + __shfl_xor_sync(0xffffffffu, send, o);
        }
        idx += up ? half : 0;
    }
#pragma unroll
    for (int o = 16 / NVAL; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    __syncthreads();
    if ((lane & (32 / NVAL - 1)) == 0) sm[warp][idx] = v[0];
    __syncthreads();
    T r = 0;
    if (threadIdx.x < NVAL)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += sm[w][threadIdx.x];
    return r;
}

// true in every thread of the last chunk block of right-hand side r
__device__ __forceinline__ bool blast_chunk(unsigned* ticket) {
    __shared__ bool am_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) am_last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
    __syncthreads();
    return am_last;
}

// sum over the chunks of value i of right-hand side r, in chunk order, by one warp
template <typename T>
__device__ __forceinline__ C2<T> bsum_chunks(const C2<T>* part_r, int i) {
    const int lane = threadIdx.x & 31;
    C2<T> acc = mk<T>(0, 0);
    for (unsigned c = lane; c < gridDim.x; c += 32) acc = cadd(acc, __ldcg(part_r + (size_t)c * RED_MAXD + i));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
    }
    return acc;
}

constexpr int BT = 256;      // threads of the batched BLAS kernels

// CH inner products of the vectors V[i0 + c], c < cnt, with w: their chunk partials
template <typename T, int CH>
__device__ __forceinline__ void bgram_chunk(const C2<T>* __restrict__ V, long ldv, int i0, int cnt,
                                            const C2<T>* __restrict__ w, long n, C2<T>* part, T (*sm)[2 * CH]) {
    const long stride = (long)gridDim.x * BT;
    C2<T> acc[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) acc[c] = mk<T>(0, 0);
    for (long e = (long)blockIdx.x * BT + threadIdx.x; e < n; e += stride) {
        const C2<T> we = w[e];
#pragma unroll
        for (int c = 0; c < CH; ++c)
            if (c < cnt) acc[c] = cfmac(V[(long)(i0 + c) * ldv + e], we, acc[c]);
    }
    const T r = bblock_sums<T, CH>(acc, sm);
    if ((int)threadIdx.x < 2 * cnt) reinterpret_cast<T*>(part + i0)[threadIdx.x] = r;
}

template <typename T>
__global__ void __launch_bounds__(BT) k_bgram(double2* __restrict__ out, long os, const C2<T>* __restrict__ V,
                                              long ldv, long vr, int nd, const int* ndd, long nds,
                                              const C2<T>* __restrict__ w, long wr, long n, C2<T>* partial,
                                              int max_chunks, unsigned* ticket, Gate g) {
    const int r = blockIdx.y;
    if (!gate_open(g, r)) return;
    __shared__ T sm8[BT / 32][16];
    __shared__ T sm2[BT / 32][4];
    int cnt = nd + (ndd ? ndd[r * nds] : 0);
    if (cnt > RED_MAXD) cnt = RED_MAXD;
    const C2<T>* Vr = V + r * vr;
    const C2<T>* wv = w + r * wr;
    C2<T>* part_r = partial + (size_t)r * max_chunks * RED_MAXD;
    C2<T>* part = part_r + (size_t)blockIdx.x * RED_MAXD;
    int i0 = 0;
    for (; cnt - i0 > 2; i0 += 8) bgram_chunk<T, 8>(Vr, ldv, i0, min(8, cnt - i0), wv, n, part, sm8);
    if (i0 < cnt) bgram_chunk<T, 2>(Vr, ldv, i0, cnt - i0, wv, n, part, sm2);
    if (blast_chunk(ticket + r)) {
        __threadfence();
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        for (int i = warp; i < cnt; i += BT / 32) {
            const C2<T> v = bsum_chunks<T>(part_r, i);
            if (lane == 0) out[r * os + i] = to_d2(v);
        }
        if (threadIdx.x == 0) ticket[r] = 0u;
    }
}

// Rows whose loads k_baxpy and k_bupdate keep in flight.  FP32 waits for memory: with one
// row at a time the updates of a 256^2 solve of 64 right-hand sides took 65 ms, with five
// and x and r of a cycle in one pass 40 ms.  FP64 is bound by its pipe and only loses warps
// to the registers (17 ms with one row, 26 ms with five).
template <typename T> constexpr int rows_ahead() { return sizeof(T) == 4 ? 5 : 1; }

template <typename T>
__global__ void __launch_bounds__(BT) k_baxpy(C2<T>* w, long wr, const C2<T>* __restrict__ V, long ldv, long vr,
                                              int nd, const int* ndd, long nds, const double2* __restrict__ coef,
                                              long cs, double sign, int zero_first, long n, double* norm2, long n2s,
                                              C2<T>* partial, int max_chunks, unsigned* ticket, Gate g) {
    const int r = blockIdx.y;
    if (!gate_open(g, r)) return;
    constexpr int BU = rows_ahead<T>();
    __shared__ C2<T> cf[RED_MAXD];
    __shared__ C2<T> sm[BT / 32];
    int cnt = nd + (ndd ? ndd[r * nds] : 0);
    if (cnt > RED_MAXD) cnt = RED_MAXD;
    for (int i = threadIdx.x; i < cnt; i += BT) {
        const double2 c = coef[r * cs + i];
        cf[i] = mk<T>((T)(sign * c.x), (T)(sign * c.y));
    }
    __syncthreads();
    const C2<T>* Vr = V + r * vr;
    C2<T>* wv = w + r * wr;
    const long stride = (long)gridDim.x * BT;
    T tacc = 0;
    for (long e = (long)blockIdx.x * BT + threadIdx.x; e < n; e += stride) {
        C2<T> a = zero_first ? mk<T>(0, 0) : wv[e];
        for (int i = 0; i < cnt; i += BU) {  // BU rows' loads in flight (a row past the last repeats it)
            C2<T> v[BU];
#pragma unroll
            for (int c = 0; c < BU; ++c) v[c] = Vr[(long)min(i + c, cnt - 1) * ldv + e];
#pragma unroll
            for (int c = 0; c < BU; ++c)
                if (i + c < cnt) a = cfma(v[c], cf[i + c], a);
        }
        wv[e] = a;
        if (norm2) tacc += a.x * a.x + a.y * a.y;
    }
    if (norm2) {
        C2<T>* part_r = partial + (size_t)r * max_chunks * RED_MAXD;
        const C2<T> v = bblock_sum<T>(mk<T>(tacc, 0), sm);
        if (threadIdx.x == 0) part_r[(size_t)blockIdx.x * RED_MAXD] = v;
        if (blast_chunk(ticket + r)) {
            __threadfence();
            if (threadIdx.x < 32) {
                const C2<T> t = bsum_chunks<T>(part_r, 0);
                if (threadIdx.x == 0) {
                    norm2[r * n2s] = (double)t.x;
                    ticket[r] = 0u;
                }
            }
        }
    }
}

// A finished cycle of cnt[r cs] steps in one pass over its basis: x = V d (or x += V d) and,
// unless r is null, r = V rho (cnt + 1 rows)
template <typename T>
__global__ void __launch_bounds__(BT) k_bupdate(C2<T>* x, long xr, C2<T>* rv, long rr, const C2<T>* __restrict__ V,
                                                long ldv, long vr, const int* __restrict__ cnt, long cs,
                                                const double2* __restrict__ d, const double2* __restrict__ rho, long ds,
                                                int accumulate, long n, Gate g) {
    const int r = blockIdx.y;
    if (!gate_open(g, r)) return;
    constexpr int BU = rows_ahead<T>();
    __shared__ C2<T> cd[RED_MAXD], cr[RED_MAXD];
    const int nd = min(cnt[r * cs], RED_MAXD - 1), rows = rv ? nd + 1 : nd;
    for (int i = threadIdx.x; i < rows; i += BT) {
        cd[i] = i < nd ? from_d2<T>(d[r * ds + i]) : mk<T>(0, 0);
        cr[i] = rv ? from_d2<T>(rho[r * ds + i]) : mk<T>(0, 0);
    }
    __syncthreads();
    const C2<T>* Vr = V + r * vr;
    for (long e = (long)blockIdx.x * BT + threadIdx.x; e < n; e += (long)gridDim.x * BT) {
        C2<T> a = accumulate ? x[r * xr + e] : mk<T>(0, 0), b = mk<T>(0, 0);
        for (int i = 0; i < rows; i += BU) {
            C2<T> v[BU];
#pragma unroll
            for (int c = 0; c < BU; ++c) v[c] = Vr[(long)min(i + c, rows - 1) * ldv + e];
#pragma unroll
            for (int c = 0; c < BU; ++c) {
                if (i + c < nd) a = cfma(v[c], cd[i + c], a);
                if (i + c < rows) b = cfma(v[c], cr[i + c], b);
            }
        }
        x[r * xr + e] = a;
        if (rv) rv[r * rr + e] = b;
    }
}

template <typename T>
__global__ void __launch_bounds__(BT) k_bnorm2(double* out, long os, const C2<T>* __restrict__ v, long vr, long n,
                                               C2<T>* partial, int max_chunks, unsigned* ticket, Gate g) {
    const int r = blockIdx.y;
    if (!gate_open(g, r)) return;
    __shared__ C2<T> sm[BT / 32];
    const C2<T>* vv = v + r * vr;
    const long stride = (long)gridDim.x * BT;
    T acc = 0;
    for (long e = (long)blockIdx.x * BT + threadIdx.x; e < n; e += stride) {
        const C2<T> a = vv[e];
        acc += a.x * a.x + a.y * a.y;
    }
    C2<T>* part_r = partial + (size_t)r * max_chunks * RED_MAXD;
    const C2<T> s = bblock_sum<T>(mk<T>(acc, 0), sm);
    if (threadIdx.x == 0) part_r[(size_t)blockIdx.x * RED_MAXD] = s;
    if (blast_chunk(ticket + r)) {
        __threadfence();
        if (threadIdx.x < 32) {
            const C2<T> t = bsum_chunks<T>(part_r, 0);
            if (threadIdx.x == 0) {
                out[r * os] = (double)t.x;
                ticket[r] = 0u;
            }
        }
    }
}

template <typename T>
__global__ void k_bscale(C2<T>* y, long yr, const C2<T>* x, long xr, const double* f, long fs, long n, Gate g) {
    const int r = blockIdx.y;
    if (!gate_open(g, r)) return;
    const T fv = (T)f[r * fs];
    C2<T>* yy = y + r * yr;
    const C2<T>* xx = x + r * xr;
    for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x)
        yy[e] = cscale(xx[e], fv);
}

template <typename Ta, typename Tb>
__global__ void k_bconvert(C2<Tb>* y, long yr, const C2<Ta>* x, long xr, long n) {
    const int r = blockIdx.y;
    C2<Tb>* yy = y + r * yr;
    const C2<Ta>* xx = x + r * xr;
    for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) {
        const C2<Ta> a = xx[e];
        yy[e] = mk<Tb>((Tb)a.x, (Tb)a.y);
    }
}

inline int chunks_for(long n, const BRed& red) {
    // an entry a thread: short vectors are bound by latency (with four, a 256^2 solve of 64
    // right-hand sides took 1% longer)
    long c = (n + BT - 1) / BT;
    if (c > red.max_chunks) c = red.max_chunks;
    if (c < 1) c = 1;
    return (int)c;
}
inline unsigned ew_chunks(long n) {
    long c = (n + 255) / 256;
    if (c > 64) c = 64;
    if (c < 1) c = 1;
    return (unsigned)c;
}

// ------------------------------------------------------ tensor-core stencil --

constexpr int NDOF = 24;
constexpr int TILE_WORDS = 64;                    // one 8 x 8 complex tile
constexpr int SITE_WORDS = 5 * 9 * TILE_WORDS;    // 5 directions x 3 x 3 tiles

template <bool F16>
__device__ __forceinline__ unsigned pack16(float re, float im) {
    if constexpr (F16) {
        const __half2 h = __floats2half2_rn(re, im);  // .x (low) = re, .y (high) = im
        return *reinterpret_cast<const unsigned*>(&h);
    } else {
        const __nv_bfloat162 h = __floats2bfloat162_rn(re, im);
        return *reinterpret_cast<const unsigned*>(&h);
    }
}
template <bool F16>
__device__ __forceinline__ float2 unpack16(unsigned u) {
    if constexpr (F16) {
        const __half2 h = *reinterpret_cast<const __half2*>(&u);
        return __half22float2(h);
    } else {
        const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&u);
        return __bfloat1622float2(h);
    }
}

template <bool F16>
__device__ __forceinline__ void mma16816(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    if constexpr (F16) {
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
            "{%0,%1,%2,%3};\n"
            : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
    } else {
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
            "{%0,%1,%2,%3};\n"
            : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
    }
}

// A fragment word of the real embedding from a complex pair (re low, im high):
// rows of real parts take (re, -im), rows of imaginary parts (im, re)
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

// FP64 -> BF16 rounded once to nearest-even: the FP64 significand is rounded at
// BF16's 8 significant bits (bit 45 of the FP64 word is the last kept one), after
// which the value converts to FP32 and to BF16 exactly (operator entries are far
// inside BF16's exponent range)
__device__ __forceinline__ unsigned short bf16_rn(double v) {
    unsigned long long u = (unsigned long long)__double_as_longlong(v);
    u += 0x00000FFFFFFFFFFFull + ((u >> 45) & 1ull);
    u &= 0xFFFFE00000000000ull;
    return __bfloat16_as_ushort(__float2bfloat16_rn((float)__longlong_as_double((long long)u)));
}

// Fragment order of a tile (output rows 8 mt + a, input columns 8 kt + c):
// word 2 (4 a + t) + e holds entry (a, t + 4 e), so the thread of group g and
// lane-in-group t loads the entries of complex row g, its rows g and g + 8 of the
// real tile, as one 8-byte vector at its lane.
template <bool F16>
__global__ void k_pack_frag(unsigned* out, const double2* __restrict__ A, long nsite) {
    const long total = nsite * SITE_WORDS;
    for (long w = (long)blockIdx.x * blockDim.x + threadIdx.x; w < total; w += (long)gridDim.x * blockDim.x) {
        const long tile = w / TILE_WORDS;
        const int q = (int)(w - tile * TILE_WORDS);
        const int e = q & 1, t = (q >> 1) & 3, a0 = q >> 3;
        const long sd = tile / 9;  // site * 5 + direction
        const int mk_ = (int)(tile - sd * 9), mt = mk_ / 3, kt = mk_ - 3 * mt;
        const int row = 8 * mt + a0, col = 8 * kt + t + 4 * e;
        const double2 v = A[(sd * NDOF + col) * NDOF + row];  // column-major block: entry (row, col)
        unsigned re, im;
        if constexpr (F16) {
            re = __half_as_ushort(__double2half(v.x));
            im = __half_as_ushort(__double2half(v.y));
        } else {
            re = bf16_rn(v.x);
            im = bf16_rn(v.y);
        }
        out[w] = (im << 16) | re;
    }
}

// Groups of G = max(1, 8 / ntiles) sites, one warp per (site, tile of 8 right-hand
// sides).  The operator of a group's sites (11.5 KB a site) is staged in shared memory
// once (cp.async), so every tile of a site reads the same copy; each warp issues all
// its neighbour-vector loads before it waits.  A CTA takes groups blockIdx.x, + gridDim.x,
// ... and stages the next one while it multiplies (WALK, two buffers): without it nothing
// was in flight during the products.  That and the
// fragment order (a third of the instructions that formed both rows of a word):
// 128 x 128 sites x 16 right-hand sides, FP16, 289 MB: 77.8 -> 68.9 us.  Where every CTA has
// one group only the kernel has no loop and no registers for it (102 instead of 127): 8
// right-hand sides on those sites 49.9 -> 48.7 us.
template <bool F16, bool RES, bool WALK>
__global__ void __launch_bounds__(256, 2) k_bstencil_mma(float2* __restrict__ Y, const float2* __restrict__ X,
                                                         const float2* __restrict__ B, long vr,
                                                         const unsigned* __restrict__ Af, int Nx, int Nt, int ntiles,
                                                         Gate g) {
    extern __shared__ uint4 bst_op[];  // [buffer] G sites x SITE_WORDS / 4
    constexpr int SITE_U4 = SITE_WORDS / 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gq = lane >> 2, t = lane & 3;
    const int nsite = Nx * Nt;
    const int G = ntiles >= 8 ? 1 : 8 / ntiles;
    const int ngroups = (nsite + G - 1) / G;
    const unsigned sbuf = (unsigned)__cvta_generic_to_shared(bst_op);
    auto stage = [&](int grp, int buf) {
        const int n = min(G, nsite - grp * G) * SITE_U4;
        const uint4* Ag = reinterpret_cast<const uint4*>(Af) + (long)grp * G * SITE_U4;
        const unsigned dst = sbuf + 16u * (unsigned)(buf * G * SITE_U4);
        for (int q = threadIdx.x; q < n; q += blockDim.x)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + 16u * q), "l"(Ag + q) : "memory");
    };
    const int ls = warp / ntiles;  // this warp's task: site ls of the group, right-hand sides r0..
    const int r0 = (warp - ls * ntiles) * NB_TILE;
    const bool live = warp < G * ntiles && __any_sync(0xffffffffu, gate_open(g, r0 + gq));
    int buf = 0;
    stage(blockIdx.x, 0);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    for (int grp = blockIdx.x; grp < ngroups; grp += gridDim.x, buf ^= 1) {
        const int s = grp * G + ls;
        const bool run = live && s < nsite;
        float2 xv[5][3][2];
        if (run) {
            const float2* Xr = X + (long)(r0 + gq) * vr;
#pragma unroll
            for (int d = 0; d < 5; ++d) {
                const float2* xn = Xr + (long)nbr_of(s, d, Nx, Nt) * NDOF;
#pragma unroll
                for (int kt = 0; kt < 3; ++kt) {
                    xv[d][kt][0] = __ldg(xn + 8 * kt + t);
                    xv[d][kt][1] = __ldg(xn + 8 * kt + t + 4);
                }
            }
        }
        if constexpr (WALK) {
            if (grp + (int)gridDim.x < ngroups) stage(grp + gridDim.x, buf ^ 1);
            asm volatile("cp.async.commit_group;\n" ::: "memory");
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        }
        __syncthreads();
        if (run) {
            float acc[3][4];
#pragma unroll
            for (int m = 0; m < 3; ++m)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[m][i] = 0.f;
            const uint2* A2 = reinterpret_cast<const uint2*>(bst_op + (buf * G + ls) * SITE_U4) + lane;
#pragma unroll
            for (int d = 0; d < 5; ++d) {
#pragma unroll
                for (int kt = 0; kt < 3; ++kt) {
                    const float2 x0 = xv[d][kt][0], x1 = xv[d][kt][1];
                    const unsigned h0 = pack16<F16>(x0.x, x0.y), h1 = pack16<F16>(x1.x, x1.y);
                    const float2 f0 = unpack16<F16>(h0), f1 = unpack16<F16>(h1);
                    const unsigned l0 = pack16<F16>(x0.x - f0.x, x0.y - f0.y),
                                   l1 = pack16<F16>(x1.x - f1.x, x1.y - f1.y);
#pragma unroll
                    for (int mt = 0; mt < 3; ++mt) {
                        const uint2 w = A2[(d * 9 + mt * 3 + kt) * (TILE_WORDS / 2)];
                        const unsigned a[4] = {embed(w.x, 0), embed(w.x, 1), embed(w.y, 0), embed(w.y, 1)};
                        mma16816<F16>(acc[mt], a, h0, h1);
                        mma16816<F16>(acc[mt], a, l0, l1);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int r = r0 + 2 * t + q;
                if (!gate_open(g, r)) continue;
                const long off = (long)r * vr + (long)s * NDOF + gq;
#pragma unroll
                for (int mt = 0; mt < 3; ++mt) {
                    float2 o = make_float2(acc[mt][q], acc[mt][2 + q]);
                    if (RES) {
                        const float2 bb = __ldg(B + off + 8 * mt);
                        o = make_float2(bb.x - o.x, bb.y - o.y);
                    }
                    Y[off + 8 * mt] = o;
                }
            }
        }
        if constexpr (!WALK) break;  // one group a CTA
        __syncthreads();  // the buffer is free for the group after the next
    }
}

}  // namespace

// ------------------------------------------------------------- launchers ----

template <typename T>
void launch_bgram(double2* out, long os, const C2<T>* V, long ldv, long vr, int nd, const int* ndd, long nds,
                  const C2<T>* w, long wr, long n, int nb, BRed red, Gate g, cudaStream_t s) {
    if (nd <= 0 && !ndd) return;
    const int ch = chunks_for(n, red);
    k_bgram<T><<<dim3(ch, nb), BT, 0, s>>>(out, os, V, ldv, vr, nd, ndd, nds, w, wr, n,
                                           reinterpret_cast<C2<T>*>(red.partial), red.max_chunks, red.ticket, g);
    count_launch();
}

template <typename T>
void launch_baxpy(C2<T>* w, long wr, const C2<T>* V, long ldv, long vr, int nd, const int* ndd, long nds,
                  const double2* coef, long cs, double sign, bool zero_first, long n, int nb, double* norm2,
                  long n2s, BRed red, Gate g, cudaStream_t s) {
    const int ch = chunks_for(n, red);
    k_baxpy<T><<<dim3(ch, nb), BT, 0, s>>>(w, wr, V, ldv, vr, nd, ndd, nds, coef, cs, sign, zero_first ? 1 : 0, n,
                                           norm2, n2s, reinterpret_cast<C2<T>*>(red.partial), red.max_chunks,
                                           red.ticket, g);
    count_launch();
}

template <typename T>
void launch_bupdate(C2<T>* x, long xr, C2<T>* r, long rr, const C2<T>* V, long ldv, long vr, const int* cnt, long cs,
                    const double2* d, const double2* rho, long ds, bool accumulate, long n, int nb, Gate g,
                    cudaStream_t s) {
    const unsigned ch = (unsigned)std::max(1L, std::min((n + BT - 1) / BT, 64L));
    k_bupdate<T><<<dim3(ch, nb), BT, 0, s>>>(x, xr, r, rr, V, ldv, vr, cnt, cs, d, rho, ds, accumulate ? 1 : 0, n, g);
    count_launch();
}

template <typename T>
void launch_bnorm2(double* out, long os, const C2<T>* v, long vr, long n, int nb, BRed red, Gate g, cudaStream_t s) {
    const int ch = chunks_for(n, red);
    k_bnorm2<T><<<dim3(ch, nb), BT, 0, s>>>(out, os, v, vr, n, reinterpret_cast<C2<T>*>(red.partial), red.max_chunks,
                                            red.ticket, g);
    count_launch();
}

template <typename T>
void launch_bscale(C2<T>* y, long yr, const C2<T>* x, long xr, const double* f, long fs, long n, int nb, Gate g,
                   cudaStream_t s) {
    k_bscale<T><<<dim3(ew_chunks(n), nb), 256, 0, s>>>(y, yr, x, xr, f, fs, n, g);
    count_launch();
}

template <typename Ta, typename Tb>
void launch_bconvert(C2<Tb>* y, long yr, const C2<Ta>* x, long xr, long n, int nb, cudaStream_t s) {
    k_bconvert<Ta, Tb><<<dim3(ew_chunks(n), nb), 256, 0, s>>>(y, yr, x, xr, n);
    count_launch();
}

void launch_pack_frag(unsigned* out, const double2* A, long nsite, bool fp16, cudaStream_t s) {
    const long total = nsite * SITE_WORDS;
    const unsigned grid = (unsigned)std::min<long>((total + 255) / 256, (long)sm_count() * 16);
    if (fp16) k_pack_frag<true><<<grid, 256, 0, s>>>(out, A, nsite);
    else k_pack_frag<false><<<grid, 256, 0, s>>>(out, A, nsite);
    count_launch();
}

void launch_bstencil_mma(float2* Y, const float2* X, const float2* B, long vr, const unsigned* Af, int Nx, int Nt,
                         int nb, bool fp16, Gate g, cudaStream_t s) {
    const int ntiles = nb / NB_TILE;
    const int G = ntiles >= 8 ? 1 : 8 / ntiles;  // sites of a group
    const long groups = ((long)Nx * Nt + G - 1) / G;
    // two CTAs an SM walk the groups with two buffers; where two buffers would leave room
    // for one CTA only (G = 8), or there is one group a CTA, a CTA takes one group
    const bool walk = G <= 4 && groups > 2L * sm_count();
    const unsigned grid = (unsigned)(walk ? 2L * sm_count() : groups);
    const size_t smem = (size_t)(walk ? 2 : 1) * G * SITE_WORDS * sizeof(unsigned);
    auto pick = [&](auto f16, auto res) {
        constexpr bool F = decltype(f16)::value, R = decltype(res)::value;
        return walk ? &k_bstencil_mma<F, R, true> : &k_bstencil_mma<F, R, false>;
    };
    const std::true_type yes{};
    const std::false_type no{};
    auto* kern = fp16 ? (B ? pick(yes, yes) : pick(yes, no)) : (B ? pick(no, yes) : pick(no, no));
    // larger than the default 48 KB when G > 4 or with two buffers
    const int mx = 8 * SITE_WORDS * (int)sizeof(unsigned);
    static std::atomic<bool> attr_set[64][8];  // once per device and kernel
    const int which = (fp16 ? 4 : 0) + (B ? 2 : 0) + (walk ? 1 : 0);
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 && !attr_set[dev][which].load())
        attr_set[dev][which].store(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, mx) ==
                                   cudaSuccess);
    kern<<<grid, 256, smem, s>>>(Y, X, B, vr, Af, Nx, Nt, ntiles, g);
    count_launch();
}

#define INST(T)                                                                                                     \
    template void launch_bgram<T>(double2*, long, const C2<T>*, long, long, int, const int*, long, const C2<T>*,    \
                                  long, long, int, BRed, Gate, cudaStream_t);                                      \
    template void launch_baxpy<T>(C2<T>*, long, const C2<T>*, long, long, int, const int*, long, const double2*,    \
                                  long, double, bool, long, int, double*, long, BRed, Gate, cudaStream_t);         \
    template void launch_bupdate<T>(C2<T>*, long, C2<T>*, long, const C2<T>*, long, long, const int*, long,         \
                                    const double2*, const double2*, long, bool, long, int, Gate, cudaStream_t);      \
    template void launch_bnorm2<T>(double*, long, const C2<T>*, long, long, int, BRed, Gate, cudaStream_t);         \
    template void launch_bscale<T>(C2<T>*, long, const C2<T>*, long, const double*, long, long, int, Gate,          \
                                   cudaStream_t);
INST(double)
INST(float)
#undef INST
template void launch_bconvert<double, float>(C2<float>*, long, const C2<double>*, long, long, int, cudaStream_t);
template void launch_bconvert<float, double>(C2<double>*, long, const C2<float>*, long, long, int, cudaStream_t);

}  // namespace mg
