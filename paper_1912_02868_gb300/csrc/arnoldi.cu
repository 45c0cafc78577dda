// The vector work of a Krylov step between two operator applies as one
// thread-block-cluster kernel, for vectors short enough that a step is bound by
// launches and reductions rather than by bytes:
//  * k_krylov_start: beta = ||f||, v_0 = f / beta and the start of the least squares
//    (norm, start and scale kernels before);
//  * k_arnoldi: CGS2 of w = V[j + 1] against V[0..j], its norm, the column's push into
//    the least squares and the normalisation (two Gram, two update, push and scale
//    kernels before, about 4 us each in a captured V-cycle);
//  * k_finish_update: the cycle's solution d and residual coefficients, x (+)= V d and
//    r = V rho (finish and two update kernels before).
// A cluster of up to 16 CTAs holds w in registers; partial sums go to every CTA's
// shared memory by distributed shared-memory stores and a cluster barrier (about
// 0.7 us), and each CTA adds them itself in rank order, so all hold the same bits.
// The arithmetic is that of the kernels it replaces: sums in the vectors' precision,
// the norm from its own pass after the second update, the least squares in FP64.
//
// Sizes: FP32 up to 131072 entries (the fine grid of 256^2), 16 a thread.  Steps in a
// captured graph, this kernel | those it replaces: 24576 entries 14.7 | 21.3 us, 65536 15.9 |
// 21.7, 131072 20.9 | 25.6 (the first two steps; over eight 29.3 | 32.1).  Longer vectors
// would spill w, and 16 SMs then bound them.  FP64 up to 16384, two a thread.  There the FP64
// pipe of 16 SMs bounds it: 4096 entries 22.2 | 24.8 us, 8192 31.4 | 25.0, 16384 41.7 | 26.8.
// But FP64 steps are launched one by one, and the host takes as long for six launches as the
// longer kernel does: FP64 solves with the limit at 16384 | 8192 | 5120 entries, 64^2 74.7 |
// 74.6 | 76.7 ms, 80 x 64 101.7 | 102.1 | 103.0, 128 x 64 131.5 | 131.5 | 131.5.
// A 256^2 mixed solve 58.8 -> 56.1 ms, a 128^2 partial solve 25.2 -> 21.1 ms, a 64^2 FP64
// solve 83.9 -> 80.4 ms.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "ks_dev.cuh"

namespace cg = cooperative_groups;

namespace mg {

namespace {

constexpr int AT = 512;        // threads a CTA
constexpr int AMAXC = 16;      // CTAs of a cluster
constexpr int ANV = 2 * KLD;   // real values of an exchange, at most

template <typename T>
struct ArnoldiSmem {
    T inbox[2][AMAXC][ANV];
    T part[ANV];
    T h[2][ANV];
    T sm[AT / 32][16];
    double scale;
    ksd::PushScratch push;
};

// sums over the CTA of the 16 real values v a thread holds (a butterfly that halves the
// values it carries, then the warps in order): thread t < 16 returns value t.  A warp
// with no entry (act false, the same for all its lanes) adds nothing and spends nothing.
template <typename T>
__device__ __forceinline__ T cta_sums16(T (&v)[16], T (*sm)[16], bool act) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (!act) {
        __syncthreads();
        if (lane < 16) sm[warp][lane] = 0;
        __syncthreads();
        T r = 0;
        if (threadIdx.x < 16)
            for (int w = 0; w < AT / 32; ++w) r += sm[w][threadIdx.x];
        return r;
    }
    int idx = 0;
#pragma unroll
    for (int half = 8, o = 16; half > 0; half >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const T send = up ? v[i] : v[i + half];
            v[i] = (up ? v[i + half] : v[i]) + __shfl_xor_sync(0xffffffffu, send, o);
        }
        idx += up ? half : 0;
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    __syncthreads();
    if (!(lane & 1)) sm[warp][idx] = v[0];
    __syncthreads();
    T r = 0;
    if (threadIdx.x < 16)
        for (int w = 0; w < AT / 32; ++w) r += sm[w][threadIdx.x];
    return r;
}
// whether this warp has an entry at all
__device__ __forceinline__ bool warp_on(long n, int nr, int me);

// S.part[0..nv) of every CTA summed in rank order into out[0..nv), the same bits in every CTA
template <typename T>
__device__ __forceinline__ void exchange(cg::cluster_group& cl, ArnoldiSmem<T>& S, int buf, int nv, T* out) {
    const int nr = (int)cl.num_blocks(), me = (int)cl.block_rank();
    __syncthreads();  // S.part complete
    for (int e = threadIdx.x; e < nr * nv; e += AT) {
        const int r = e / nv, v = e - r * nv;
        *cl.map_shared_rank(&S.inbox[buf][me][v], r) = S.part[v];
    }
    if (nr > 1) cl.sync();
    else __syncthreads();
    for (int e = threadIdx.x; e < 4 * ((nv + 7) & ~7); e += AT) {  // whole warps: 8 values each
        const int v = e >> 2, q = e & 3;
        T s = 0;
        if (v < nv)
            for (int r = q; r < nr; r += 4) s += S.inbox[buf][r][v];
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (q == 0 && v < nv) out[v] = s;
    }
    __syncthreads();
}

// entry i of this thread (n: none): CTA `me` of nr takes whole warps' worth of
// consecutive entries
__device__ __forceinline__ long elem(long n, int nr, int me, int i) {
    const long chunk = ((n + nr - 1) / nr + 31) & ~31L, t = (long)i * AT + threadIdx.x;
    return t < chunk ? me * chunk + t : n;
}

__device__ __forceinline__ bool warp_on(long n, int nr, int me) {
    const long chunk = ((n + nr - 1) / nr + 31) & ~31L, t = threadIdx.x & ~31;
    return t < chunk && me * chunk + t < n;
}

// S.part[2 c], [2 c + 1] = the CTA's partial of conj(V[c]) . w, c < nd
template <typename T, int E>
__device__ __forceinline__ void gram_regs(ArnoldiSmem<T>& S, const C2<T>* __restrict__ V, long n, int nd,
                                          const C2<T> (&w)[E], int nr, int me) {
    for (int c0 = 0; c0 < nd; c0 += 8) {
        C2<T> acc[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = mk<T>(0, 0);
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const long e = elem(n, nr, me, i);
            if (e >= n) break;
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c0 + c < nd) acc[c] = cfmac(V[(long)(c0 + c) * n + e], w[i], acc[c]);
        }
        T v[16];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            v[2 * c] = acc[c].x;
            v[2 * c + 1] = acc[c].y;
        }
        const T r = cta_sums16<T>(v, S.sm, warp_on(n, nr, me));
        if (threadIdx.x < 16 && c0 + (int)threadIdx.x / 2 < nd) S.part[2 * c0 + threadIdx.x] = r;
    }
}

// sum over the cluster of |w|^2
template <typename T, int E>
__device__ __forceinline__ T norm2_regs(cg::cluster_group& cl, ArnoldiSmem<T>& S, const C2<T> (&w)[E], long n,
                                        int buf, T* out) {
    T v[16] = {};
#pragma unroll
    for (int i = 0; i < E; ++i) v[0] += w[i].x * w[i].x + w[i].y * w[i].y;  // (zero past the vector's end)
    const T r = cta_sums16<T>(v, S.sm, warp_on(n, (int)cl.num_blocks(), (int)cl.block_rank()));
    if (threadIdx.x == 0) S.part[0] = r;
    exchange<T>(cl, S, buf, 1, out);
    return out[0];
}

template <typename T, int E>
__global__ void __launch_bounds__(AT) k_arnoldi(C2<T>* __restrict__ V, long n, int j, KState* ks, Gate g) {
    extern __shared__ __align__(16) unsigned char arn_smem[];
    ArnoldiSmem<T>& S = *reinterpret_cast<ArnoldiSmem<T>*>(arn_smem);
    if (!gate_open(g)) return;  // the same for every CTA: only this kernel's end changes it, after its barriers
    cg::cluster_group cl = cg::this_cluster();
    const int nr = (int)cl.num_blocks(), me = (int)cl.block_rank(), nd = j + 1;
    C2<T>* const wv = V + (long)nd * n;
    C2<T> w[E];
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const long e = elem(n, nr, me, i);
        w[i] = e < n ? wv[e] : mk<T>(0, 0);
    }
    if (nr > 1) cl.sync();  // every CTA of the cluster runs before the first remote store
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {  // CGS2
        gram_regs<T, E>(S, V, n, nd, w, nr, me);
        exchange<T>(cl, S, pass, 2 * nd, S.h[pass]);
        const C2<T>* h = reinterpret_cast<const C2<T>*>(S.h[pass]);
        for (int c = 0; c < nd; ++c) {
            const C2<T> hc = h[c];
#pragma unroll
            for (int i = 0; i < E; ++i) {
                const long e = elem(n, nr, me, i);
                if (e < n) w[i] = cfma(V[(long)c * n + e], mk<T>(-hc.x, -hc.y), w[i]);
            }
        }
    }
    __shared__ T nrm;
    const double hn2 = (double)norm2_regs<T, E>(cl, S, w, n, 0, &nrm);
    if (threadIdx.x == 0) S.scale = hn2 > 0.0 ? rsqrt(hn2) : 1.0;
    __syncthreads();
    const T sc = (T)S.scale;
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const long e = elem(n, nr, me, i);
        if (e < n) wv[e] = cscale(w[i], sc);
    }
    if (me == 0 && threadIdx.x < 32) {
        for (int c = threadIdx.x; c < nd; c += 32) {
            ks->hA[c] = make_double2((double)S.h[0][2 * c], (double)S.h[0][2 * c + 1]);
            ks->hB[c] = make_double2((double)S.h[1][2 * c], (double)S.h[1][2 * c + 1]);
        }
        if (threadIdx.x == 0) ks->hn2 = hn2;
        __syncwarp();
        ksd::ks_push_warp(ks, j, S.push);
    }
    if (nr > 1) cl.sync();  // no CTA leaves while others may still write its shared memory
}

template <typename T, int E>
__global__ void __launch_bounds__(AT) k_krylov_start(C2<T>* __restrict__ v0, const C2<T>* __restrict__ f, long n,
                                                     KState* ks) {
    extern __shared__ __align__(16) unsigned char arn_smem[];
    ArnoldiSmem<T>& S = *reinterpret_cast<ArnoldiSmem<T>*>(arn_smem);
    cg::cluster_group cl = cg::this_cluster();
    const int nr = (int)cl.num_blocks(), me = (int)cl.block_rank();
    C2<T> w[E];
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const long e = elem(n, nr, me, i);
        w[i] = e < n ? f[e] : mk<T>(0, 0);
    }
    if (nr > 1) cl.sync();
    __shared__ T nrm;
    const double b2 = (double)norm2_regs<T, E>(cl, S, w, n, 0, &nrm);
    if (threadIdx.x == 0) S.scale = b2 > 0.0 ? rsqrt(b2) : 0.0;
    __syncthreads();
    const T sc = (T)S.scale;
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const long e = elem(n, nr, me, i);
        if (e < n) v0[e] = cscale(w[i], sc);
    }
    if (me == 0 && threadIdx.x < 32) ksd::ks_start_dev(ks, b2, 0.0, b2);
    if (nr > 1) cl.sync();
}

constexpr int FU_STEPS = 8;  // longest cycle of k_finish_update

// every block finishes the small least squares itself; block 0 also stores the results
template <typename T>
__global__ void __launch_bounds__(256) k_finish_update(C2<T>* __restrict__ x, C2<T>* __restrict__ r,
                                                       const C2<T>* __restrict__ V, long n, KState* ks, int accumulate) {
    __shared__ double2 Rs[FU_STEPS * (FU_STEPS + 1) / 2], ds[FU_STEPS], rhos[FU_STEPS + 1];
    __shared__ C2<T> dc[FU_STEPS], rc[FU_STEPS + 1];
    const int jj = ks->j;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        ksd::load_upper(Rs, ks->R, jj, lane, 32);
        __syncwarp();
        ksd::solve_upper(Rs, ks->g, ds, jj, blockIdx.x == 0 ? &ks->err : nullptr);
        double part = 0.0;
        if (lane <= jj) {
            double2 acc = ks->c[lane];
            for (int l = 0; l < jj; ++l) acc = csub(acc, cmul(ks->H[lane + KLD * l], ds[l]));
            rhos[lane] = acc;
            rc[lane] = from_d2<T>(acc);
            part = acc.x * acc.x + acc.y * acc.y;
        }
        if (lane < jj) dc[lane] = from_d2<T>(ds[lane]);
        if (blockIdx.x == 0) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
            __syncwarp();
            if (lane < jj) ks->d[lane] = ds[lane];
            for (int i = lane; i < KLD; i += 32) ks->rho[i] = i <= jj ? rhos[i] : make_double2(0.0, 0.0);
            if (lane == 0) ks->res = sqrt(part);
        }
    }
    __syncthreads();
    for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) {
        C2<T> a = accumulate ? x[e] : mk<T>(0, 0), b = mk<T>(0, 0);
#pragma unroll 4
        for (int i = 0; i <= jj; ++i) {
            if (i == jj && !r) break;
            const C2<T> v = V[(long)i * n + e];
            if (i < jj) a = cfma(v, dc[i], a);
            if (r) b = cfma(v, rc[i], b);
        }
        x[e] = a;
        if (r) r[e] = b;
    }
}

struct Shape {
    int ctas, e;
};
// The CTAs of the cluster and entries a thread (0: too long).  FP32: at most eight entries
// a thread before the cluster grows.  FP64: about 96 entries a CTA, so that the FP64
// instructions spread over SMs as early as a cluster barrier costs less than they do.
template <typename T>
Shape shape_of(long n) {
    if (std::is_same<T, double>::value) {
        int c = 1;
        while (c < AMAXC && n > 96L * c) c <<= 1;
        for (int e = 1; e <= 2; e <<= 1)
            if (n <= (long)c * AT * e) return {c, e};
        return {0, 0};
    }
    for (int c = 1; c <= AMAXC; c <<= 1)
        for (int e = 1; e <= (c == AMAXC ? 16 : 8); e <<= 1)
            if (n <= (long)c * AT * e) return {c, e};
    return {0, 0};
}

template <typename F>
bool configure(F* f, size_t smem) {
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = AMAXC;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(AMAXC);
    cfg.blockDim = dim3(AT);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, f, &cfg) != cudaSuccess || nc < 1) {
        (void)cudaGetLastError();
        return false;
    }
    return true;
}

// one-time set-up of both kernels with E elements a thread on the current device
template <typename T, int E>
bool ready() {
    static std::mutex mu;
    static signed char state[16] = {};  // 0: not tried, 1: ready, -1: not available
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 16) {
        (void)cudaGetLastError();
        return false;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (state[dev] == 0)
        state[dev] = configure(&k_arnoldi<T, E>, sizeof(ArnoldiSmem<T>)) &&
                             configure(&k_krylov_start<T, E>, sizeof(ArnoldiSmem<T>))
                         ? 1
                         : -1;
    return state[dev] == 1;
}

template <typename F, typename... A>
void launch(F* f, int ctas, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(AT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, f, args...);
    count_launch();
}

// F(integral_constant<E>) for the shape's E
template <typename T, typename F>
bool with_shape(long n, F&& f) {
    const Shape sh = shape_of<T>(n);
    switch (sh.e) {
        case 1: return ready<T, 1>() && (f(std::integral_constant<int, 1>{}, sh.ctas), true);
        case 2: return ready<T, 2>() && (f(std::integral_constant<int, 2>{}, sh.ctas), true);
        default: break;
    }
    if constexpr (std::is_same<T, float>::value) {
        switch (sh.e) {
            case 4: return ready<T, 4>() && (f(std::integral_constant<int, 4>{}, sh.ctas), true);
            case 8: return ready<T, 8>() && (f(std::integral_constant<int, 8>{}, sh.ctas), true);
            case 16: return ready<T, 16>() && (f(std::integral_constant<int, 16>{}, sh.ctas), true);
            default: break;
        }
    }
    return false;
}

}  // namespace

template <typename T>
bool launch_arnoldi(C2<T>* V, long n, int j, KState* ks, Gate g, cudaStream_t s) {
    return with_shape<T>(n, [&](auto e, int ctas) {
        launch(&k_arnoldi<T, decltype(e)::value>, ctas, sizeof(ArnoldiSmem<T>), s, V, n, j, ks, g);
    });
}
template <typename T>
bool launch_krylov_start(C2<T>* v0, const C2<T>* f, long n, KState* ks, cudaStream_t s) {
    return with_shape<T>(n, [&](auto e, int ctas) {
        launch(&k_krylov_start<T, decltype(e)::value>, ctas, sizeof(ArnoldiSmem<T>), s, v0, f, n, ks);
    });
}
template <typename T>
bool launch_finish_update(C2<T>* x, C2<T>* r, const C2<T>* V, long n, int steps, KState* ks, bool accumulate,
                          cudaStream_t s) {
    if (steps > FU_STEPS) return false;
    const long blocks = std::min<long>((n + 255) / 256, 2L * sm_count());
    k_finish_update<T><<<(unsigned)blocks, 256, 0, s>>>(x, r, V, n, ks, accumulate ? 1 : 0);
    count_launch();
    return true;
}

template bool launch_arnoldi<double>(double2*, long, int, KState*, Gate, cudaStream_t);
template bool launch_arnoldi<float>(float2*, long, int, KState*, Gate, cudaStream_t);
template bool launch_krylov_start<double>(double2*, const double2*, long, KState*, cudaStream_t);
template bool launch_krylov_start<float>(float2*, const float2*, long, KState*, cudaStream_t);
template bool launch_finish_update<double>(double2*, double2*, const double2*, long, int, KState*, bool, cudaStream_t);
template bool launch_finish_update<float>(float2*, float2*, const float2*, long, int, KState*, bool, cudaStream_t);

}  // namespace mg
