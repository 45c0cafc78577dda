// Restriction P^+ and prolongation P between grids (Section 2: the columns of
// P are the chirally doubled near-null vectors, blocked on 4^2 sites and
// orthonormalised per block and chirality).
//
// Q[B][c][j][l][a]: coarse site B, chirality c, vector j < 12, finer site
// l = lx + 4 lt of the 4x4 block, dof a < h of chirality c at that site
// (h = 1 on the fine grid, 12 on the intermediate grid).  Coarse dof k = 12c + j.
//   restrict:  v^[B][k]           = sum_{l,a} conj(Q[B][c][j][l][a]) v[s(B,l)][c h + a]
//   prolong:   v[s(B,l)][c h + a] = sum_j Q[B][c][j][l][a] v^[B][12 c + j]
#include "batch.cuh"

namespace mg {

namespace {

constexpr int NV = 12;      // near-null vectors per chirality
constexpr int BL = 4;       // block extent
constexpr int BS = BL * BL; // sites per block

template <typename T> struct alignas(16) CPair {  // two adjacent complex entries
    C2<T> a, b;
};
template <typename T>
__device__ __forceinline__ CPair<T> ld_pair(const C2<T>* p) {
    return *reinterpret_cast<const CPair<T>*>(p);
}
template <typename T>
__device__ __forceinline__ void add_xor(C2<T>& v, int o) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
}
// the same from a caller's vector, which may start on any entry (AL: on a pair)
template <typename T, bool AL>
__device__ __forceinline__ CPair<T> ld_pair_of(const C2<T>* p) {
    if constexpr (AL) return ld_pair<T>(p);
    CPair<T> q;
    q.a = p[0];
    q.b = p[1];
    return q;
}
// bit i: gate of right-hand side r0 + i open, i < cnt <= 32 (one load round for all)
__device__ __forceinline__ unsigned gates_of(const Gate& g, int r0, int cnt) {
    const int lane = threadIdx.x & 31;
    return __ballot_sync(0xffffffffu, lane < cnt && gate_open(g, r0 + lane));
}

constexpr int RST_RHS = 16;  // right-hand sides that one read of P serves

// Restriction.  The bytes are P's (16 h complex entries per coarse dof, once per
// launch for up to RST_RHS right-hand sides) and the vectors'; the kernel is bound by
// how many of P's loads are in flight, so a lane issues all of its share of a coarse
// site's columns at once, 16 bytes each, and keeps them in registers for every
// right-hand side.  One warp per column with the h, site and row indices divided out
// per element kept two loads in flight and half the lanes idle at h = 1.
//
// Fine grid (h = 1): one warp per coarse site.  Lane (kk, m) = (lane / 8, lane % 8)
// holds entries 2m, 2m + 1 of columns 4 it + kk, it < 6, and sums them over its
// eight lanes; lane m = it stores.
template <typename T, bool AL>
__global__ void __launch_bounds__(256) k_restrict_fine(C2<T>* __restrict__ vc, const C2<T>* __restrict__ v,
                                                       const C2<T>* __restrict__ Q, int NxF, int nc, int nb, long cr,
                                                       long fr, Gate g) {
    const int lane = threadIdx.x & 31, B = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int r0 = blockIdx.y * RST_RHS, cnt = min(RST_RHS, nb - r0);
    if (B >= nc) return;
    const unsigned on = gates_of(g, r0, cnt);
    if (!on) return;
    const int NxC = NxF / BL, bx = B % NxC, bt = B / NxC;
    const int kk = lane >> 3, m = lane & 7;
    const C2<T>* q = Q + ((long)B * 2 * NV + kk) * BS + 2 * m;
    CPair<T> qv[6];
#pragma unroll
    for (int it = 0; it < 6; ++it) qv[it] = ld_pair<T>(q + it * 4 * BS);
    const long fs = (long)(bt * BL + m / 2) * NxF + bx * BL + 2 * (m & 1);
#pragma unroll 2
    for (int i = 0; i < cnt; ++i) {
        if (!((on >> i) & 1u)) continue;
        const C2<T>* vr = v + (long)(r0 + i) * fr + 2 * fs;
        const CPair<T> s0 = ld_pair_of<T, AL>(vr), s1 = ld_pair_of<T, AL>(vr + 2);  // both spins of sites 2m, 2m + 1
        C2<T> out = mk<T>(0, 0);
#pragma unroll
        for (int it = 0; it < 6; ++it) {
            C2<T> acc = cfmac(qv[it].a, it < 3 ? s0.a : s0.b, mk<T>(0, 0));
            acc = cfmac(qv[it].b, it < 3 ? s1.a : s1.b, acc);
            add_xor<T>(acc, 1);
            add_xor<T>(acc, 2);
            add_xor<T>(acc, 4);
            if (m == it) out = acc;
        }
        if (m < 6) vc[(long)(r0 + i) * cr + (long)B * 2 * NV + 4 * m + kk] = out;
    }
}

// Intermediate grid (h = 12): one CTA of eight warps per coarse site, three columns
// of one chirality per warp, six entries of each (three adjacent pairs, 32 lanes
// apart) per lane.
template <typename T, bool AL>
__global__ void __launch_bounds__(256) k_restrict_int(C2<T>* __restrict__ vc, const C2<T>* __restrict__ v,
                                                      const C2<T>* __restrict__ Q, int NxF, int nb, long cr, long fr,
                                                      Gate g) {
    constexpr int H = NV, LEN = BS * H;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, B = blockIdx.x;
    const int r0 = blockIdx.y * RST_RHS, cnt = min(RST_RHS, nb - r0);
    const unsigned on = gates_of(g, r0, cnt);
    if (!on) return;
    const int NxC = NxF / BL, bx = B % NxC, bt = B / NxC;
    const int k0 = 3 * warp, c = k0 / NV;
    const C2<T>* q = Q + ((long)B * 2 * NV + k0) * LEN;
    CPair<T> qv[3][3];
    long off[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const int e = 2 * (lane + 32 * p), l = e / H, a = e - l * H;
#pragma unroll
        for (int j = 0; j < 3; ++j) qv[j][p] = ld_pair<T>(q + (long)j * LEN + e);
        off[p] = ((long)(bt * BL + l / BL) * NxF + bx * BL + (l % BL)) * 2 * H + c * H + a;
    }
#pragma unroll 2
    for (int i = 0; i < cnt; ++i) {
        if (!((on >> i) & 1u)) continue;
        const C2<T>* vr = v + (long)(r0 + i) * fr;
        CPair<T> x[3];
#pragma unroll
        for (int p = 0; p < 3; ++p) x[p] = ld_pair_of<T, AL>(vr + off[p]);
        C2<T> acc[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            acc[j] = mk<T>(0, 0);
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                acc[j] = cfmac(qv[j][p].a, x[p].a, acc[j]);
                acc[j] = cfmac(qv[j][p].b, x[p].b, acc[j]);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < 3; ++j) add_xor<T>(acc[j], o);
        if (lane < 3) vc[(long)(r0 + i) * cr + (long)B * 2 * NV + k0 + lane] = lane == 0 ? acc[0] : lane == 1 ? acc[1] : acc[2];
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_prolong(C2<T>* __restrict__ v, const C2<T>* __restrict__ vc,
                                                 const C2<T>* __restrict__ Q, int NxF, int NtF, int h, int accumulate,
                                                 long fr, long cr, Gate g) {
    const int rb = blockIdx.y;
    if (!gate_open(g, rb)) return;
    v += rb * fr;
    vc += rb * cr;
    const long nf = (long)NxF * NtF * 2 * h;
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nf) return;
    const long fs = e / (2 * h);
    const int r = (int)(e - fs * 2 * h);
    const int c = r / h, a = r - c * h;
    const int xf = (int)(fs % NxF), tf = (int)(fs / NxF);
    const int B = (tf / BL) * (NxF / BL) + xf / BL;
    const int l = (xf % BL) + BL * (tf % BL);
    const C2<T>* q = Q + (((long)B * 2 * NV + c * NV) * BS + l) * h + a;
    const C2<T>* w = vc + (long)B * 2 * NV + c * NV;
    C2<T> acc = accumulate ? v[e] : mk<T>(0, 0);
#pragma unroll
    for (int j = 0; j < NV; ++j) acc = cfma(q[(long)j * BS * h], w[j], acc);
    v[e] = acc;
}

}  // namespace

template <typename T>
void launch_brestrict(C2<T>* coarse, long cr, const C2<T>* fine, long fr, const C2<T>* Q, int NxF, int NtF, int h,
                      int nb, Gate g, cudaStream_t s) {
    const int nc = (NxF / BL) * (NtF / BL);
    const unsigned ry = (unsigned)((nb + RST_RHS - 1) / RST_RHS);
    // the two coarsenings of the hierarchy: h = 1 on the fine grid, NV on the intermediate one
    const bool al = reinterpret_cast<size_t>(fine) % 16 == 0 && (nb == 1 || fr % 2 == 0);
    const dim3 gf((nc + 7) / 8, ry), gi(nc, ry);
    if (h == 1) {
        if (al) k_restrict_fine<T, true><<<gf, 256, 0, s>>>(coarse, fine, Q, NxF, nc, nb, cr, fr, g);
        else k_restrict_fine<T, false><<<gf, 256, 0, s>>>(coarse, fine, Q, NxF, nc, nb, cr, fr, g);
    } else {
        if (al) k_restrict_int<T, true><<<gi, 256, 0, s>>>(coarse, fine, Q, NxF, nb, cr, fr, g);
        else k_restrict_int<T, false><<<gi, 256, 0, s>>>(coarse, fine, Q, NxF, nb, cr, fr, g);
    }
    count_launch();
}

template <typename T>
void launch_bprolong(C2<T>* fine, long fr, const C2<T>* coarse, long cr, const C2<T>* Q, int NxF, int NtF, int h,
                     bool accumulate, int nb, Gate g, cudaStream_t s) {
    const long nf = (long)NxF * NtF * 2 * h;
    k_prolong<T><<<dim3(nblocks(nf, 256), nb), 256, 0, s>>>(fine, coarse, Q, NxF, NtF, h, accumulate ? 1 : 0, fr, cr,
                                                              g);
    count_launch();
}

template <typename T>
void launch_restrict(C2<T>* coarse, const C2<T>* fine, const C2<T>* Q, int NxF, int NtF, int h, Gate g,
                     cudaStream_t s) {
    launch_brestrict<T>(coarse, 0, fine, 0, Q, NxF, NtF, h, 1, g, s);
}

template <typename T>
void launch_prolong(C2<T>* fine, const C2<T>* coarse, const C2<T>* Q, int NxF, int NtF, int h, bool accumulate,
                    Gate g, cudaStream_t s) {
    launch_bprolong<T>(fine, 0, coarse, 0, Q, NxF, NtF, h, accumulate, 1, g, s);
}

template void launch_restrict<double>(C2<double>*, const C2<double>*, const C2<double>*, int, int, int, Gate,
                                      cudaStream_t);
template void launch_restrict<float>(C2<float>*, const C2<float>*, const C2<float>*, int, int, int, Gate,
                                     cudaStream_t);
template void launch_prolong<double>(C2<double>*, const C2<double>*, const C2<double>*, int, int, int, bool, Gate,
                                     cudaStream_t);
template void launch_prolong<float>(C2<float>*, const C2<float>*, const C2<float>*, int, int, int, bool, Gate,
                                    cudaStream_t);
template void launch_brestrict<double>(C2<double>*, long, const C2<double>*, long, const C2<double>*, int, int, int,
                                       int, Gate, cudaStream_t);
template void launch_brestrict<float>(C2<float>*, long, const C2<float>*, long, const C2<float>*, int, int, int, int,
                                      Gate, cudaStream_t);
template void launch_bprolong<double>(C2<double>*, long, const C2<double>*, long, const C2<double>*, int, int, int,
                                      bool, int, Gate, cudaStream_t);
template void launch_bprolong<float>(C2<float>*, long, const C2<float>*, long, const C2<float>*, int, int, int, bool,
                                     int, Gate, cudaStream_t);

}  // namespace mg
