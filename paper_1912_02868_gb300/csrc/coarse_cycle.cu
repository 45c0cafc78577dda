// The Arnoldi steps of a batched coarse GMRES-Proj cycle with the newest work on chip:
// the cycle kernel of coarse_block.cu for chunks of at most 16 coarse sites.  Same
// method, same split into site chunks x tiles of eight right-hand sides with the whole
// grid resident (cooperative launch), same sums in chunk order in every CTA.
//
// A step there was the latency of one CTA's chain (48.6 us at 256^2 x 64 right-hand
// sides, 35 us with a single tile): one warp a right-hand side walked its basis rows in
// L2 three times, a site's operator was staged per step, and three count-and-generation
// barriers of 3 us separated the phases.  Here:
//  * Two warps a right-hand side, w in registers (E pairs of entries a thread) through
//    both orthogonalisations; the loads of four rows are in flight at once.
//  * A CTA's first `srows` basis rows stay in its shared memory (8 of 21 at 14 sites a
//    chunk): rows are read four times a step, the operator once, so the rows get the
//    space and the operator streams from L2 one direction ahead.  (With half of that
//    space for operator buffers the step was slower.)  An entry is always read by the
//    thread that wrote it, so rows need no barrier.
//  * The sums of a pass travel as words that carry their step's tag (as in
//    coarse_tc.cu's grid form): a reader polls the partials themselves, so an exchange
//    is one store and one load, without barrier, fence or counter.  The new basis row is
//    published by one release flag a CTA; the stop decisions by one tagged word a tile,
//    made from one FP64 dot product while the rotations run on a warp nobody waits for.
// A cycle of 20 steps, 256^2 x 64, alone and cold: 788 -> 572 us (28.6 us a step); with the
// projection and finish around it 48.4 -> 34.5 us a step; the whole solve 511 -> 418 ms.
// Still latencies (L2 at 16% of its rate): apply 7 us (an L2 round is 0.6 us), the two
// passes over the rows 3.4 and 6.7 us, their exchanges 3 us each, the update 2.8 us.
//
// Reuse of the exchange words: a CTA writes partials of step j + 1 only after every
// CTA of the tile has raised its flag of step j, which it does after reading all
// partials and the gate word of step j; it raises the flag of step j + 1 only after a
// second-pass sum of step j + 1, to which every CTA contributed after waiting for the
// flags of step j.  Tags are the launch's base (advanced by k_cb_gate_init) + step + 1.
//
// Every wait polls at most `spin` times; one that gives up sets *err and the CTA's fault
// flag, after which its waits poll once, so every launch ends.  Decisions that guard a
// CTA barrier are read from shared memory, the same for all its warps.
#include <algorithm>
#include <type_traits>

#include "coarse_block_dev.cuh"

namespace mg {

using namespace cbdev;

namespace {

constexpr int RW = 2 * NB_TILE;          // row warps: two a right-hand side
constexpr int XM = (RW + 1) * 32;        // and one that decides and polls: they meet at main_sync
constexpr int XT = XM + 32;              // and one that rotates columns in the background
constexpr int XMAXSPC = RW;              // a warp applies one site
constexpr int XMAXCH = 128;              // chunks

struct CBXSmem {
    CBPush p;
    float2 h[2][NB_TILE][MAXI + 3];  // reduced products of the two passes, zero up to the next multiple of four
    float nrm[NB_TILE];
    float part[RW][64];          // a warp's sums, real and imaginary parts
    unsigned live[2];            // right-hand sides that take the step, by its parity
    // chunk 0: the left null vector t of each right-hand side's Arnoldi matrix, |t|^2, the
    // squares of the cycle's first residual and of its tolerance, and the decisions
    double2 t[NB_TILE][MAXI + 1];
    double nu[NB_TILE], beta2[NB_TILE], tol2[NB_TILE];
    int stop[NB_TILE];
    int cmd;                     // column for the background warp to rotate (-1: none follows)
    unsigned cmd_mask;
    int fault;
#ifdef CB_PHASE_CLOCKS
    unsigned clk;
#endif
};

__device__ __forceinline__ void st_tagged(ulonglong2* p, float x, float y, unsigned tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};\n" ::"l"(p), "l"(t | __float_as_uint(x)),
                 "l"(t | __float_as_uint(y))
                 : "memory");
}
__device__ __forceinline__ ulonglong2 ld_tagged(const ulonglong2* p) {
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];\n" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}
// the two warps of right-hand side rl of the tile
__device__ __forceinline__ void pair_sync(int rl) { asm volatile("bar.sync %0, 64;\n" ::"r"(1 + rl) : "memory"); }
__device__ __forceinline__ void main_sync() { asm volatile("bar.sync 10, %0;\n" ::"n"(XM) : "memory"); }
// the deciding warp and the background warp of chunk 0: a column is ready, it is rotated
__device__ __forceinline__ void ready_sync() { asm volatile("bar.sync 11, 64;\n" ::: "memory"); }
__device__ __forceinline__ void done_sync() { asm volatile("bar.sync 12, 64;\n" ::: "memory"); }
__device__ __forceinline__ void row_sync() { asm volatile("bar.sync 9, %0;\n" ::"n"(RW * 32) : "memory"); }

__device__ __forceinline__ long polls(const int* fault, long spin) {
    return *reinterpret_cast<const volatile int*>(fault) ? 1 : spin;
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

// Where a thread's basis rows lie: the pairs p0 + 64 u, u < E, of entries of right-hand
// side r on the chunk.  A pair past the chunk's end (zero in w) reads the last one.
template <int E>
struct Rows {
    const float2* sm;    // row 0 in shared memory (of this thread's right-hand side)
    const float2* gl;    // row 0 in global memory (of this chunk and right-hand side)
    long srow, grow;     // their row strides
    int srows;
    int p[E];
    unsigned on;         // bit u: pair u is in the chunk
    __device__ __forceinline__ const float4* row(int i) const {
        return reinterpret_cast<const float4*>(i < srows ? sm + i * srow : gl + i * grow);
    }
};

// part[2 i], [2 i + 1] = this warp's sums of conj(row i) w, i < nd, and nn as value nd.
// Packed FMAs: (Re Re, Im Im) and (Re Im, Im Re) of row and w are summed as they lie.
template <int E>
__device__ __forceinline__ void warp_gram(const Rows<E>& R, int nd, const float4 (&w)[E], bool norm, float nn,
                                          float* part) {
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int g0 = 0; g0 < nd + (norm ? 1 : 0); g0 += 8) {
        float v[16];
#pragma unroll
        for (int c0 = 0; c0 < 8; c0 += 4) {
            float4 x[4][E];  // four rows' loads in flight (a row past the last repeats it)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float4* p = R.row(min(g0 + c0 + c, nd - 1));
#pragma unroll
                for (int u = 0; u < E; ++u) x[c][u] = p[R.p[u]];
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float2 p = make_float2(0.f, 0.f), q = p;
#pragma unroll
                for (int u = 0; u < E; ++u) {
                    p = fma2(make_float2(x[c][u].x, x[c][u].y), make_float2(w[u].x, w[u].y), p);
                    q = fma2(make_float2(x[c][u].x, x[c][u].y), make_float2(w[u].y, w[u].x), q);
                    p = fma2(make_float2(x[c][u].z, x[c][u].w), make_float2(w[u].z, w[u].w), p);
                    q = fma2(make_float2(x[c][u].z, x[c][u].w), make_float2(w[u].w, w[u].z), q);
                }
                v[2 * (c0 + c)] = norm && g0 + c0 + c == nd ? nn : p.x + p.y;
                v[2 * (c0 + c) + 1] = q.x - q.y;
            }
        }
        int idx = 0;
#pragma unroll
        for (int half = 8, o = 16; half > 0; half >>= 1, o >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int i = 0; i < half; ++i) {
                const float send = up ? v[i] : v[i + half];
                v[i] = (up ? v[i + half] : v[i]) + __shfl_xor_sync(0xffffffffu, send, o);
            }
            idx += up ? half : 0;
        }
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        if (!(lane & 1)) part[2 * g0 + idx] = v[0];
    }
}

// The pair's sums to the chunk's words of gp[value][chunk], then h[i] (and *nrm, value nd)
// = the sums over all chunks: eight lanes a value, each over every eighth chunk in
// order, then a fixed tree.  false when a wait gave up.
__device__ __forceinline__ bool pair_exchange(CBXSmem& S, ulonglong2* gp, int c, int nch, int nd, bool norm, int rl,
                                              int half, unsigned tag, long spin, float2* h, float* nrm) {
    const int lane = threadIdx.x & 31, q = half * 32 + lane, nv = nd + (norm ? 1 : 0);
    pair_sync(rl);
    if (q < nv)
        st_tagged(gp + (long)q * nch + c, S.part[rl][2 * q] + S.part[rl + NB_TILE][2 * q],
                  S.part[rl][2 * q + 1] + S.part[rl + NB_TILE][2 * q + 1], tag);
    const int grp = q >> 3, l = lane & 7;
    bool ok = true;
#pragma unroll 1
    for (int i0 = 0; i0 < max(nv, (nd + 3) & ~3); i0 += 16) {
        float2 s[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll 1
        for (int c0 = 0; c0 < nch; c0 += 32) {
            ulonglong2 x[2][4];
            unsigned wait = 0;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                x[b >> 2][b & 3] = make_ulonglong2(0, 0);
                if (i0 + 8 * (b >> 2) + grp < nv && c0 + 8 * (b & 3) + l < nch) wait |= 1u << b;
            }
            for (long it = 0; wait && it < spin; ++it) {
#pragma unroll
                for (int b = 0; b < 8; ++b)
                    if ((wait >> b) & 1u)
                        x[b >> 2][b & 3] = ld_tagged(gp + (long)(i0 + 8 * (b >> 2) + grp) * nch + c0 + 8 * (b & 3) + l);
#pragma unroll
                for (int b = 0; b < 8; ++b) {
                    const ulonglong2 y = x[b >> 2][b & 3];
                    if ((unsigned)(y.x >> 32) == tag && (unsigned)(y.y >> 32) == tag) wait &= ~(1u << b);
                }
            }
            ok = ok && wait == 0;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                s[b >> 2].x += __uint_as_float((unsigned)x[b >> 2][b & 3].x);
                s[b >> 2].y += __uint_as_float((unsigned)x[b >> 2][b & 3].y);
            }
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 2; ++k) {
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                s[k].x += __shfl_xor_sync(0xffffffffu, s[k].x, o);
                s[k].y += __shfl_xor_sync(0xffffffffu, s[k].y, o);
            }
            const int i = i0 + 8 * k + grp;
            if (l == 0 && i < ((nd + 3) & ~3)) h[i] = i < nd ? s[k] : make_float2(0.f, 0.f);
            if (l == 0 && norm && i == nd) *nrm = s[k].x;
        }
    }
    pair_sync(rl);
    return ok;
}

// w -= sum_i row i h[i] (h is zero from nd to the next multiple of four)
template <int E>
__device__ __forceinline__ void subtract(const Rows<E>& R, int nd, const float2* h, float4 (&w)[E]) {
#pragma unroll 1
    for (int i = 0; i < nd; i += 4) {
        float4 x[4][E];  // four rows' loads in flight (a row past the last repeats it)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float4* r = R.row(min(i + c, nd - 1));
#pragma unroll
            for (int u = 0; u < E; ++u) x[c][u] = r[R.p[u]];
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float2 k = h[i + c];
#pragma unroll
            for (int u = 0; u < E; ++u) {
                w[u].x -= x[c][u].x * k.x - x[c][u].y * k.y;
                w[u].y -= x[c][u].x * k.y + x[c][u].y * k.x;
                w[u].z -= x[c][u].z * k.x - x[c][u].w * k.y;
                w[u].w -= x[c][u].z * k.y + x[c][u].w * k.x;
            }
        }
    }
#pragma unroll
    for (int u = 0; u < E; ++u)
        if (!((R.on >> u) & 1u)) w[u] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// w = A v_jh at site s0 + warp for the tile's right-hand sides, into ws[rl][site 24 + row].
// sv: row jh of the chunk in shared memory (null: not there), for neighbours in the chunk.
template <bool F16>
__device__ __forceinline__ void apply_site(const CBArgs& a, int jh, int r0, int s0, int ns, const float2* sv, float2* ws,
                                           int wst) {
    const int lane = threadIdx.x & 31, ls = threadIdx.x >> 5;
    if (ls >= ns) return;
    const int gq = lane >> 2, t = lane & 3;
    const int s = s0 + ls;
    const float2* Xr = a.V + (long)jh * a.row + (long)(r0 + gq) * a.n;
    const uint2* A2 = reinterpret_cast<const uint2*>(a.Af) + (long)s * (SITE_WORDS / 2) + lane;
    float acc[3][4];
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[m][i] = 0.f;
    float2 x[2][3][2];
    uint2 aw[2][3][3];
    auto load = [&](int d, int k) {
        const int u = nbr_of(s, d, a.Nx, a.Nt), lu = u - s0;
        if (sv && lu >= 0 && lu < ns) {
            const float2* xn = sv + gq * wst + lu * NDOF + t;
#pragma unroll
            for (int kt = 0; kt < 3; ++kt) {
                x[k][kt][0] = xn[8 * kt];
                x[k][kt][1] = xn[8 * kt + 4];
            }
        } else {
            const float2* xn = Xr + (long)u * NDOF + t;
#pragma unroll
            for (int kt = 0; kt < 3; ++kt) {
                x[k][kt][0] = __ldcg(xn + 8 * kt);
                x[k][kt][1] = __ldcg(xn + 8 * kt + 4);
            }
        }
#pragma unroll
        for (int kt = 0; kt < 3; ++kt)
#pragma unroll
            for (int m = 0; m < 3; ++m) aw[k][kt][m] = __ldg(A2 + (d * 9 + m * 3 + kt) * (TILE_WORDS / 2));
    };
    load(0, 0);
#pragma unroll
    for (int d = 0; d < 5; ++d) {
        if (d < 4) load(d + 1, (d + 1) & 1);  // in flight during this direction's products
        const int k = d & 1;
#pragma unroll
        for (int kt = 0; kt < 3; ++kt) {
            const float2 x0 = x[k][kt][0], x1 = x[k][kt][1];
            const unsigned h0 = pk<F16>(x0.x, x0.y), h1 = pk<F16>(x1.x, x1.y);
            const float2 f0 = upk<F16>(h0), f1 = upk<F16>(h1);
            const unsigned l0 = pk<F16>(x0.x - f0.x, x0.y - f0.y), l1 = pk<F16>(x1.x - f1.x, x1.y - f1.y);
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const uint2 w = aw[k][kt][m];
                const unsigned av[4] = {embed(w.x, 0), embed(w.x, 1), embed(w.y, 0), embed(w.y, 1)};
                mma<F16>(acc[m], av, h0, h1);
                mma<F16>(acc[m], av, l0, l1);
            }
        }
    }
    // lane (gq, t) holds output row gq of each tile for right-hand sides 2t, 2t + 1
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        float2* o = ws + 2 * t * wst + ls * NDOF + 8 * m + gq;
        o[0] = make_float2(acc[m][0], acc[m][2]);
        o[wst] = make_float2(acc[m][1], acc[m][3]);
    }
}

#ifdef CB_PHASE_CLOCKS
__device__ unsigned cbx_clock_launches = 0;
#define CBX_STAMP(k)                            \
    do {                                        \
        if (clk && threadIdx.x == 0) {          \
            const long long now = clock64();    \
            acc_t[k] += now - t_prev;           \
            t_prev = now;                       \
        }                                       \
    } while (0)
#else
#define CBX_STAMP(k) \
    do {             \
    } while (0)
#endif

// stride of a right-hand side in the shared-memory rows: two entries of padding spread
// the apply's stores over the banks
__host__ __device__ constexpr int row_stride(int spc) { return spc * NDOF + 2; }

template <bool F16, int E>
__global__ void __launch_bounds__(XT, 1) k_cb_chunk(const __grid_constant__ CBArgs a, int ms, long spin, int* err) {
    extern __shared__ __align__(16) unsigned char cbx_smem[];
    CBXSmem& S = *reinterpret_cast<CBXSmem*>(cbx_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tile = blockIdx.y, r0 = tile * NB_TILE, c = blockIdx.x, nch = a.nchunks;
    const int s0 = c * a.spc, ns = min(a.spc, a.Nx * a.Nt - s0);
    const int wst = row_stride(a.spc), srow = NB_TILE * wst;
    float2* const ws = reinterpret_cast<float2*>(cbx_smem + sizeof(CBXSmem));
    float2* const Vc = ws + srow;
    const bool rw = warp < RW;
    const int rl = warp & (NB_TILE - 1), half = warp >> 3, r = r0 + rl;
    const unsigned base = __ldcg(a.epoch);
    unsigned long long* const gword = a.gword + tile;
    unsigned* const flags = a.flags + tile * XMAXCH;
    ulonglong2* const gp1 = a.t1 + (long)r * CB_PB * nch;
    ulonglong2* const gp2 = a.t2 + (long)r * CB_PB * nch;
    float2* const Vr = a.V + (long)r * a.n + (long)s0 * NDOF;
    Rows<E> R;
    R.sm = Vc + rl * wst;
    R.gl = Vr;
    R.srow = srow;
    R.grow = a.row;
    R.srows = a.srows;
    R.on = 0;
    const int np = ns * NDOF / 2;
#pragma unroll
    for (int u = 0; u < E; ++u) {
        const int p = half * 32 + lane + 64 * u;
        R.p[u] = min(p, np - 1);
        R.on |= (p < np ? 1u : 0u) << u;
    }
    auto give_up = [&] {
        *reinterpret_cast<volatile int*>(&S.fault) = 1;
        atomicExch(err, 1);
    };
#ifdef CB_PHASE_CLOCKS
    if (tid == 0) S.clk = (c == 1 && tile == 0) ? (atomicAdd(&cbx_clock_launches, 1u) & 63u) == 20u : 0;
    __syncthreads();
    const bool clk = S.clk != 0;
    long long acc_t[8] = {0, 0, 0, 0, 0, 0, 0, 0}, t_prev = clock64();
    int steps = 0;
#endif
    if (tid == 0) S.fault = 0;
    __syncthreads();
    if (a.probe && tid == 0) {  // test probe: a wait that nothing ends gives up
        const volatile unsigned* never = a.bar + 2 * (NB_MAX / NB_TILE);
        long it = 0;
        while (*never == 0u) {
            if (++it > spin) {
                give_up();
                break;
            }
            __nanosleep(32);
        }
    }
    if (warp == RW) {
        if (c == 0 && lane < NB_TILE) {  // the least squares as the cycle's start left it
            const KState* ks = a.ks + r0 + lane;
            for (int i = 0; i <= MSMAX; ++i) S.p.g[lane][i] = ks->g[i];
            S.p.tol[lane] = ks->tol_abs;
            S.t[lane][0] = make_double2(1.0, 0.0);
            S.nu[lane] = 1.0;
            S.beta2[lane] = ks->beta * ks->beta;
            S.tol2[lane] = ks->tol_abs * ks->tol_abs;
        }
        const unsigned m = gate_mask(a.gbuf, r0, 0);
        if (lane == 0) S.live[0] = m;
    } else if (rw && a.srows > 0) {
        for (int p = half * 32 + lane; p < np; p += 64)
            reinterpret_cast<float4*>(Vc + rl * wst)[p] = __ldcg(reinterpret_cast<const float4*>(Vr) + p);
    }
    __syncthreads();
    if (warp > RW) {  // the background warp: R, g and the rotations of each column
        if (c == 0)
            while (true) {
                ready_sync();
                const int jc = S.cmd;
                if (jc < 0) break;
                if (lane < NB_TILE && ((S.cmd_mask >> lane) & 1u))
                    push_cycle(a, S.p, lane, r0 + lane, jc, S.stop[lane]);
                done_sync();
            }
        return;
    }
    // Chunk 0's deciding warp, after step jc of the right-hand sides in `took`: which go on.
    // Column jc is orthogonal to conj(t), so t grows by one entry a column, t_{jc+1} =
    // -(sum_i t_i h_i) / h_{jc+1}, and the least-squares residual is beta / |t|: four lanes a
    // right-hand side and one dot product, where the rotations are a chain of 12 FP64
    // instructions an earlier column (10 us at the end of a cycle, and every CTA waits).
    bool sent = false;
    auto close_column = [&](int jc, unsigned took) {
        if (sent) done_sync();  // the background warp has rotated the column before
        const int q = lane >> 2, f = lane & 3;
        const bool on = (took >> q) & 1u;
        double2 dot = make_double2(0.0, 0.0);
        if (on) {
            push_column_entries(S.p, q, jc, S.h[1][q], f, 4);
            for (int i = f; i <= jc; i += 4) dot = cfma(S.t[q][i], S.p.col[q][i], dot);
        }
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
            dot.x += __shfl_xor_sync(0xffffffffu, dot.x, o);
            dot.y += __shfl_xor_sync(0xffffffffu, dot.y, o);
        }
        bool go = false;
        if (on && f == 0) {
            const double hn = (double)S.p.hn[q];
            bool conv = true;
            if (hn != 0.0) {
                const double inv = 1.0 / hn;
                const double2 tn = make_double2(-dot.x * inv, -dot.y * inv);
                const double nu = S.nu[q] + tn.x * tn.x + tn.y * tn.y;
                S.t[q][jc + 1] = tn;
                S.nu[q] = nu;
                conv = S.beta2[q] <= S.tol2[q] * nu;
                go = !conv;
            }
            S.stop[q] = conv ? 1 : 0;
        }
        const unsigned b = __ballot_sync(0xffffffffu, go);
        unsigned m = 0;
#pragma unroll
        for (int i = 0; i < NB_TILE; ++i) m |= ((b >> (4 * i)) & 1u) << i;
        if (lane == 0) {
            S.cmd = jc;
            S.cmd_mask = took;
        }
        __syncwarp();
        sent = true;
        return m;
    };
    unsigned spec = S.live[0];  // right-hand sides that took the last step (the first: that take it)
    int jh = 0;
    for (; jh < ms && spec; ++jh) {
        const unsigned tag = base + (unsigned)jh + 1u;
        const int nd = jh + 1;
        float4 w[E];
        if (rw) {
            // w = A v_jh and its first products, for every right-hand side that took the step
            // before; the stop decisions of that step come in meanwhile
            apply_site<F16>(a, jh, r0, s0, ns, jh < a.srows ? Vc + (long)jh * srow : nullptr, ws, wst);
            row_sync();
            CBX_STAMP(0);
            if ((spec >> rl) & 1u) {
#pragma unroll
                for (int u = 0; u < E; ++u)
                    w[u] = (R.on >> u) & 1u ? reinterpret_cast<const float4*>(ws + rl * wst)[R.p[u]]
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
                warp_gram<E>(R, nd, w, false, 0.f, S.part[warp]);
                CBX_STAMP(1);
                if (!pair_exchange(S, gp1, c, nch, nd, false, rl, half, tag, polls(&S.fault, spin), S.h[0][rl], nullptr))
                    give_up();
            }
        } else if (jh > 0) {
            unsigned m = 0;
            if (c == 0) {
                m = close_column(jh - 1, spec);
                if (lane == 0)
                    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;\n" ::"l"(gword),
                                 "l"(((unsigned long long)tag << 32) | m)
                                 : "memory");
                ready_sync();
            } else if (lane == 0) {
                const long n = polls(&S.fault, spin);
                long it = 0;
                for (; it < n; ++it) {
                    unsigned long long v;
                    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];\n" : "=l"(v) : "l"(gword) : "memory");
                    if ((unsigned)(v >> 32) == tag) {
                        m = (unsigned)v;
                        break;
                    }
                }
                if (it == n) give_up();
            }
            if (lane == 0) S.live[jh & 1] = m;
        }
        main_sync();
        CBX_STAMP(2);
        const unsigned live = S.live[jh & 1];
        if (!live) break;
        if (rw && ((live >> rl) & 1u)) {
            // (chunk 0's deciding warp has read the last step's S.p.h1: it came to the barrier after)
            if (c == 0 && half == 0 && lane < nd) S.p.h1[rl][lane] = S.h[0][rl][lane];
            subtract<E>(R, nd, S.h[0][rl], w);
            float nn = 0.f;
#pragma unroll
            for (int u = 0; u < E; ++u)
                nn += w[u].x * w[u].x + w[u].y * w[u].y + w[u].z * w[u].z + w[u].w * w[u].w;
            warp_gram<E>(R, nd, w, true, nn, S.part[warp]);
            CBX_STAMP(3);
            if (!pair_exchange(S, gp2, c, nch, nd, true, rl, half, tag, polls(&S.fault, spin), S.h[1][rl], &S.nrm[rl]))
                give_up();
            CBX_STAMP(4);
            // h_{j+1,j} = ||w - V h2|| = sqrt(||w||^2 - ||h2||^2) (the basis is orthonormal)
            const float2 h2 = lane < nd ? S.h[1][rl][lane] : make_float2(0.f, 0.f);
            float h2n = h2.x * h2.x + h2.y * h2.y;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) h2n += __shfl_xor_sync(0xffffffffu, h2n, o);
            const float hn = sqrtf(fmaxf(S.nrm[rl] - h2n, 0.f)), inv = hn > 0.f ? 1.f / hn : 0.f;
            if (lane == 0 && half == 0) S.p.hn[rl] = hn;
            subtract<E>(R, nd, S.h[1][rl], w);
#pragma unroll
            for (int u = 0; u < E; ++u)
                if ((R.on >> u) & 1u) {
                    const float4 v = make_float4(w[u].x * inv, w[u].y * inv, w[u].z * inv, w[u].w * inv);
                    reinterpret_cast<float4*>(Vr + (long)nd * a.row)[R.p[u]] = v;
                    if (nd < a.srows) reinterpret_cast<float4*>(Vc + (long)nd * srow + rl * wst)[R.p[u]] = v;
                }
        }
        CBX_STAMP(5);
        // publish v_{j+1}: the CTA's stores precede its flag, and every flag this CTA's loads
        main_sync();
        if (tid == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;\n" ::"l"(flags + c), "r"(tag) : "memory");
        if (warp == RW) {
            const long n = polls(&S.fault, spin);
            for (int q = lane; q < nch; q += 32) {
                long it = 0;
                for (; it < n; ++it) {
                    unsigned v;
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(flags + q) : "memory");
                    if (v == tag) break;
                }
                if (it == n) give_up();
            }
        }
        main_sync();
        CBX_STAMP(6);
        spec = live;
#ifdef CB_PHASE_CLOCKS
        ++steps;
#endif
    }
    // the last step's column, when the loop ran to the cycle length (after an early exit every
    // column has been closed: the exit follows the phase that did it)
    if (warp == RW && c == 0) {
        if (jh == ms) {
            close_column(ms - 1, spec);
            ready_sync();
        }
        if (sent) done_sync();
        if (lane == 0) S.cmd = -1;
        __syncwarp();
        ready_sync();
    }
#ifdef CB_PHASE_CLOCKS
    if (clk && tid == 0 && steps > 0)
        printf("cb_chunk clocks/step over %d steps, %d chunks of %d, %d rows: apply %lld, gram1 %lld, exch1+gate %lld, "
               "upd+gram2 %lld, exch2 %lld, update %lld, publish %lld\n",
               steps, nch, a.spc, a.srows, acc_t[0] / steps, acc_t[1] / steps, acc_t[2] / steps, acc_t[3] / steps,
               acc_t[4] / steps, acc_t[5] / steps, acc_t[6] / steps);
#endif
}

// E of the kernel: pairs of entries a thread
bool two_pairs(int spc) { return spc * NDOF / 2 <= 64 * 2; }
size_t row_bytes(int spc) { return (size_t)NB_TILE * row_stride(spc) * sizeof(float2); }

const void* kernel_of(bool fp16, int spc) {
    if (two_pairs(spc)) return fp16 ? (const void*)&k_cb_chunk<true, 2> : (const void*)&k_cb_chunk<false, 2>;
    return fp16 ? (const void*)&k_cb_chunk<true, 3> : (const void*)&k_cb_chunk<false, 3>;
}

// shared memory beside the basis rows
size_t fixed_smem(int spc) { return sizeof(CBXSmem) + row_bytes(spc); }
size_t chunk_smem(const CBArgs& a) { return fixed_smem(a.spc) + (size_t)a.srows * row_bytes(a.spc); }

}  // namespace

size_t cb_chunk_words(int nbp) { return (size_t)nbp * CB_PB * XMAXCH; }
int cb_chunk_flags() { return NB_MAX / NB_TILE * XMAXCH; }

// Chunks of at most 16 sites, one CTA an SM.  As few sites as fill the SMs, but not so few
// that the exchanges, which grow with the chunks, cost more than the rows: at least 1/32
// of the grid.
bool cb_geometry_chunk(CBArgs& a, long nsite, int nbp, bool fp16) {
    const long ntiles = nbp / NB_TILE, sms = sm_count();
    if (ntiles > sms) return false;
    const long per = sms / ntiles;  // chunks of a tile that are resident at once
    long spc = std::max((nsite + per - 1) / per, std::min((long)XMAXSPC, (nsite + 31) / 32));
    spc = std::max(spc, std::min(nsite, 4L));
    if (spc > XMAXSPC) return false;
    const long nch = (nsite + spc - 1) / spc;
    if (nch > XMAXCH) return false;
    a.spc = (int)spc;
    a.nchunks = (int)nch;
    a.nbp = nbp;
    a.coop = 2;
    int dev = 0, smax = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smax, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    const long room = (long)smax - (long)fixed_smem(a.spc);
    if (room < 0) return false;
    a.srows = (int)std::min<long>(room / (long)row_bytes(a.spc), MAXI);
    const void* f = kernel_of(fp16, a.spc);
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smax) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, XT, chunk_smem(a)) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return per_sm >= 1;
}

mg_status launch_cb_chunk(const CBArgs& a, int ms, bool fp16, long spin, int* err, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.gridDim = dim3(a.nchunks, a.nbp / NB_TILE);
    cfg.blockDim = dim3(XT);
    cfg.dynamicSmemBytes = chunk_smem(a);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const bool e2 = two_pairs(a.spc);
    if (fp16) {
        if (e2) MG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_cb_chunk<true, 2>, a, ms, spin, err));
        else MG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_cb_chunk<true, 3>, a, ms, spin, err));
    } else {
        if (e2) MG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_cb_chunk<false, 2>, a, ms, spin, err));
        else MG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_cb_chunk<false, 3>, a, ms, spin, err));
    }
    count_launch();
    return MG_OK;
}

}  // namespace mg
