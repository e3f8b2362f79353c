// fold.cu -- folded nets: the first pass over a ReLU net whose neurons mostly keep
// their sign in the box.
//
// Over one query's box (s pixels moved by at most k grey levels) a hidden neuron
// whose potential cannot cross zero acts linearly: its output change is its
// potential's change ("pos") or 0 ("neg"). Folding those neurons into the weights
// leaves, exactly, a small net on the box: every kept potential is
//     du_n = sum_p A_np x_p + sum_m C_nm dh_m,     x_p = dv_p / 255  (Eq. 1)
// over the s pixel changes and the output changes dh_m of the few neurons of
// earlier layers whose sign can change (the "nodes"). Only nodes and outputs need
// evaluating: every other neuron's sign is known to be the unperturbed image's at
// every point, so it adds neither a sign change nor a sign tie (Sec. III-B).
//
//   k_pro_layer (prologue.cu)  rows A, C as FP32 pairs, layer by layer, from the rows
//                 of the layer below; B_n >= |du_n| over the box; the class
//                 ("pos"/"neg" when |ub_n| > B_n, its error and the tie band)
//   k_fold_pack   per query: the rows of nodes and outputs as FP32 in groups of 4,
//                 their error bounds; D and the margin of the unperturbed image
//   k_fold        the first pass: 4 points per thread, FP32 on CUDA cores
//   k_fold64      the points it left undecided, a warp each, the same rows in FP64:
//                 every result by its definition, sign ties and margin ties included
// and what lies within its error of the tie band's edge (about 1e-12 around tau)
// goes to the FP64 pass on the whole net. A query with more than kFoldMax nodes is not folded; its general
// passes run instead (they return at once for folded queries).
//
// Error of k_fold, constant per node (u = 2^-24, K sources, M_n = sum_k |c_nk| bound
// of source k): the FMA chain and the roundings of c and x give at most
// (K + 4) u M_n, the sources' own errors sum |C_nm| e_m, the rows' fer_n, the
// base potential |fl(ub) - ub| + eub, its addition u (|ub| + B_n). Their sum e_n
// bounds both |u_n - exact| and, since the ReLU is 1-Lipschitz, |dh_n - exact|.
// A sign is certain when |u_n| > e_n + 2 tau, a margin when it exceeds e_D + e_o + 2 tau.
//
// Why: on boxes of a few pixels moved by up to 15 grey levels about 1 % of the neurons
// can change sign, so a point costs a few hundred multiply-adds instead of the 268 k of
// 784-512-512-10 (or 2.1 M of 784-1024-1024-1024-10), in FP32 with a bound of about
// 1e-7 instead of a 16-bit screen's 1e-4..1e-2, and almost no point is left for a
// second pass. Whole calls, before and after: 784-512-512-10, s = 6, k = 7 (11.4 M
// points near the boundary) 28.7 -> 1.5 ms; 784-1024x3-10, s = 4, k = 15 with coverage
// 191 -> 4.3 ms; 784-300-100-10, s = 5, k = 9 in an L2 ball 27.7 -> 0.52 ms.
#include "dev.cuh"
#include "dfloat.cuh"
#include "launch.h"

#include <cfloat>

namespace vbmc {
namespace {

constexpr int FT = 256;          // threads of k_fold
constexpr int FW = FT / 32;
constexpr int FP = 128;          // points per warp block: 4 per lane, 32 apart
constexpr int kFoldSm = 1024;    // coefficient entries kept in shared memory (larger: through L1)
constexpr int kPairW = kFoldMax / 32;

// Nodes and packed coefficients by layer: layer l's n[l] rows (nodes; l = L: the
// outputs, class D first) have src(l) = s + cb[l] columns; entry off[l] + g src + k
// of fc32 holds column k of the rows 4 g .. 4 g + 3.
struct FoldShape {
    int n[kMaxL + 1], cb[kMaxL + 1], off[kMaxL + 1];
    int entries, nodes;
};

__device__ void fold_shape(const NetView& net, const QueryView& Q, FoldShape& f) {
    int cb = 0, off = 0;
    for (int l = 1; l <= net.L; ++l) {
        const int n = l < net.L ? Q.fst[2 + l] : net.dims[l];
        f.n[l] = n;
        f.cb[l] = cb;
        f.off[l] = off;
        off += ((n + 3) >> 2) * (Q.s + cb);
        if (l < net.L) cb += n;
    }
    f.entries = off;
    f.nodes = cb;
}

// Output held by row i of the output layer: D first, then the others in order.
__device__ __forceinline__ int out_of_row(int i, int D) { return i == 0 ? D : (i <= D ? i - 1 : i); }

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__global__ void __launch_bounds__(256) k_fold_pack(NetView net, QueryView* qs, unsigned long long* unfolded) {
    __shared__ FoldShape f;
    __shared__ float eh[kFoldMax], eh64[kFoldMax], eo[kFoldOut];
    __shared__ int D_s;
    QueryView& Q = qs[blockIdx.x];
    if (!Q.fold || Q.fst[1] || (Q.cnt->err & DERR_PIXELS)) {
        if (threadIdx.x == 0 && unfolded) atomicAdd(unfolded, 1ull);
        return;
    }
    const int L = net.L, HL = net.dims[L], offL = net.noff[L], s = Q.s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {  // D: the largest output, the lowest index among equals; HL <= 32
        const double y = lane < HL ? Q.ub[offL + lane] : -DBL_MAX;
        const double top = warp_max(y);
        const int D = __ffs(__ballot_sync(0xffffffffu, lane < HL && y == top)) - 1;
        const double mx = warp_max(lane == D ? -DBL_MAX : y);
        if (lane == 0) {
            D_s = D;
            Q.cnt->D = D;
            Q.cnt->base_margin = Q.prop == PROP_THRESHOLD ? fmax(top - Q.V, Q.V - mx) : top - mx;
        }
    } else if (threadIdx.x == 32) {
        fold_shape(net, Q, f);
    }
    __syncthreads();
    const int D = D_s;
    auto neuron = [&](int l, int i) { return l < L ? Q.fnode[f.cb[l] + i] : offL + out_of_row(i, D); };
    for (int e = threadIdx.x; e < f.entries; e += blockDim.x) {
        int l = L;
        while (e < f.off[l]) --l;  // layers without rows have the offset of the next one
        const int src = s + f.cb[l], n = f.n[l], g = (e - f.off[l]) / src, k = e - f.off[l] - g * src;
        float c[4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
            c[r] = 4 * g + r < n ? Q.fco[(size_t)neuron(l, 4 * g + r) * Q.fstride + k].x : 0.f;
        Q.fc32[e] = make_float4(c[0], c[1], c[2], c[3]);
    }
    // error bounds (FP32, rounded up), layer by layer: a warp per row, its lanes over the sources
    const float tau2 = __double2float_ru(2.0 * kTau);
    for (int l = 1; l <= L; ++l) {
        const int cb = f.cb[l];
        for (int i = warp; i < f.n[l]; i += blockDim.x / 32) {
            const int nn = neuron(l, i);
            const float2* row = Q.fco + (size_t)nn * Q.fstride;
            float M = 0.f, pr = 0.f, pr64 = 0.f;
            for (int k = lane; k < s + cb; k += 32) {
                const float w = abs_up(row[k]);
                if (k < s) {
                    M = __fmaf_ru(w, Q.fx[k], M);
                } else {
                    M = __fmaf_ru(w, __fadd_ru(Q.fbd[Q.fnode[k - s]], eh[k - s]), M);
                    pr = __fmaf_ru(w, eh[k - s], pr);
                    pr64 = __fmaf_ru(w, eh64[k - s], pr64);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                M = __fadd_ru(M, __shfl_xor_sync(0xffffffffu, M, o));
                pr = __fadd_ru(pr, __shfl_xor_sync(0xffffffffu, pr, o));
                pr64 = __fadd_ru(pr64, __shfl_xor_sync(0xffffffffu, pr64, o));
            }
            if (lane) continue;
            const double ub = Q.ub[nn];
            const float ub32 = (float)ub, B = Q.fbd[nn], fer = Q.fer[nn], eub = Q.fhe[nn].y;
            const float mag = __fadd_ru(__fadd_ru(fabsf(ub32), B), 1e-30f);
            const float ed = __fadd_ru(__fmaf_ru((float)(s + cb + 5) * 0x1p-24f, M, pr), __fadd_ru(fer, 1e-37f));
            float e = __fadd_ru(__fadd_ru(ed, __double2float_ru(fabs((double)ub32 - ub))), eub);
            e = __fmaf_ru(0x1.01p-24f, __fadd_ru(mag, ed), e);
            // the same in FP64 (u = 2^-53; x_p = dv_p / 255 rounds once, the rows' pairs are exact in it)
            const float e64 = __fmaf_ru(0x1p-51f, mag, __fadd_ru(__fmaf_ru((float)(s + cb + 6) * 0x1p-53f, M, pr64),
                                                                 __fadd_ru(fer, eub)));
            Q.fe64[l < L ? cb + i : kFoldMax + i] = e64;
            const float e2 = __fadd_ru(e, tau2);
            const float thr = fabs(ub) < kTau ? INFINITY : e2;  // a base tie: every sign is a tie
            if (l < L) {
                eh[cb + i] = e;
                eh64[cb + i] = e64;
                Q.fk32[cb + i] = make_float4(ub32, ub >= 0.0 ? 0.f : ub32, ub >= 0.0 ? -ub32 : 0.f, thr);
            } else {
                eo[i] = __fmaf_ru(0x1.01p-23f, mag, e);
                Q.fk32[kFoldMax + i] = make_float4(ub32, e2, 0.f, thr);
            }
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < HL; i += blockDim.x)
        Q.fk32[kFoldMax + i].z = __fadd_ru(__fadd_ru(eo[0], eo[i]), tau2);
    if (threadIdx.x == 0) {
        Q.fst[0] = 1;
        Q.cnt->folded = 1;
    }
}

struct FoldSm {
    float4 co[2 * kFoldSm];              // entry k: (c0, c0, c1, c1), (c2, c2, c3, c3): operands of paired FMAs
    float4 kc[kFoldMax + kFoldOut];      // fk32
    float xs[kMaxS * kMaxR];             // [s][R] fl(dv / 255)
    uint32_t prow[kFoldMax][kPairW];     // SS pairs of node m with row i of the next layer
    unsigned char hit[kFoldMax + kFoldOut];  // nodes and outputs that changed sign at some point
    FoldShape f;
    int D;
    unsigned long long g;
};

struct FoldAcc {  // per warp, over a segment of one query
    unsigned long long adv = 0, first = ~0ull, pts = 0;
};

// 128 consecutive points from tb (a multiple of 32) of query Q.
template <bool SM>
__device__ __forceinline__ void fold_points(const NetView& net, const QueryView& Q, FoldSm& S,
                                            unsigned long long tb, unsigned long long tend, FoldAcc& acc,
                                            const Queue& out, int out_level, unsigned q) {
    const int lane = threadIdx.x & 31;
    const int s = Q.s, R = Q.R, L = net.L;
    const bool cov = Q.flip != nullptr;
    float4 src[kMaxS + kFoldMax];  // sources of the 4 points: pixel changes, then node changes
    unsigned vm = 0;               // bit i: point tb + 32 i + lane is checked
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const unsigned long long t = tb + 32 * i + lane;
        vm |= (unsigned)(t >= Q.lo && t < tend) << i;
    }
    if (!Q.filter && tend + FP <= 0xFFFFFFFFull) {
        // t / R by the 32-bit reciprocal floor((2^32 - 1) / R): at most one too small
        unsigned tt[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) tt[i] = (unsigned)tb + 32 * i + lane;
        const unsigned Ru = (unsigned)R, inv = 0xFFFFFFFFu / Ru;
        for (int p = s - 1; p >= 0; --p) {
            float x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                unsigned d = __umulhi(tt[i], inv), r = tt[i] - d * Ru;
                if (r >= Ru) {
                    r -= Ru;
                    ++d;
                }
                tt[i] = d;
                x[i] = S.xs[p * R + (int)r];
            }
            src[p] = make_float4(x[0], x[1], x[2], x[3]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned long long t = tb + 32 * i + lane;
            int d[kMaxS];
            decode_digits((vm >> i) & 1u ? t : Q.lo, s, R, d);
            if (Q.filter && !in_filter(Q, d)) vm &= ~(1u << i);  // L2 ball / shell
            for (int p = 0; p < s; ++p) reinterpret_cast<float*>(&src[p])[i] = S.xs[p * R + d[p]];
        }
        if (Q.filter) {
            int c = __popc(vm);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
            acc.pts += (unsigned)c;
        }
    }
    unsigned unc = 0, und = 0, neg = 0;  // bits per point: a sign not certain; margin undecided / negative
    unsigned da = 0, db = 0, oa = 0, ob = 15u;  // Eq. 11: sides of V
    unsigned cprev = 0, iprev = 0, ccur = 0, icur = 0;  // per point (bytes): changes of a layer, the last one
    float yD[4] = {0.f, 0.f, 0.f, 0.f};
    const bool eq11 = Q.prop == PROP_THRESHOLD;
    for (int l = 1; l <= L; ++l) {
        const int n = S.f.n[l], cb = S.f.cb[l], ns = s + cb;
        cprev = ccur;
        iprev = icur;
        ccur = 0;
        for (int g = 0; 4 * g < n; ++g) {
            float2 a[4][2];
#pragma unroll
            for (int e = 0; e < 4; ++e) a[e][0] = a[e][1] = make_float2(0.f, 0.f);
            const int e0 = S.f.off[l] + g * ns;
#pragma unroll 4
            for (int k = 0; k < ns; ++k) {
                const float4 v = src[k];
                float4 c01, c23;
                if (SM) {
                    c01 = S.co[2 * (e0 + k)];
                    c23 = S.co[2 * (e0 + k) + 1];
                } else {
                    const float4 c = __ldg(&Q.fc32[e0 + k]);
                    c01 = make_float4(c.x, c.x, c.y, c.y);
                    c23 = make_float4(c.z, c.z, c.w, c.w);
                }
                const float2 v0 = make_float2(v.x, v.y), v1 = make_float2(v.z, v.w);
                a[0][0] = __ffma2_rn(make_float2(c01.x, c01.y), v0, a[0][0]);
                a[0][1] = __ffma2_rn(make_float2(c01.x, c01.y), v1, a[0][1]);
                a[1][0] = __ffma2_rn(make_float2(c01.z, c01.w), v0, a[1][0]);
                a[1][1] = __ffma2_rn(make_float2(c01.z, c01.w), v1, a[1][1]);
                a[2][0] = __ffma2_rn(make_float2(c23.x, c23.y), v0, a[2][0]);
                a[2][1] = __ffma2_rn(make_float2(c23.x, c23.y), v1, a[2][1]);
                a[3][0] = __ffma2_rn(make_float2(c23.z, c23.w), v0, a[3][0]);
                a[3][1] = __ffma2_rn(make_float2(c23.z, c23.w), v1, a[3][1]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = 4 * g + e;
                if (i >= n) break;
                const float du[4] = {a[e][0].x, a[e][0].y, a[e][1].x, a[e][1].y};
                const int at = l < L ? cb + i : kFoldMax + i;
                const float4 kk = S.kc[at];
                float u[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) u[j] = kk.x + du[j];
                if (l < L) {
                    src[s + cb + i] = make_float4(fmaxf(du[0] + kk.y, kk.z), fmaxf(du[1] + kk.y, kk.z),
                                                  fmaxf(du[2] + kk.y, kk.z), fmaxf(du[3] + kk.y, kk.z));
                } else if (i == 0) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) yD[j] = u[j];
                }
                if (l == L) {
                    if (eq11) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int sd = thr_side(u[j], (float)Q.V, kk.y);
                            if (i == 0) {
                                da |= (unsigned)(sd > 0) << j;
                                db |= (unsigned)(sd < 0) << j;
                            } else {
                                oa |= (unsigned)(sd > 0) << j;
                                if (!(sd < 0)) ob &= ~(1u << j);
                            }
                        }
                    } else if (i > 0) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float diff = yD[j] - u[j];
                            neg |= (unsigned)(diff < -kk.z) << j;
                            und |= (unsigned)!(fabsf(diff) > kk.z) << j;
                        }
                    }
                }
                if (cov) {
                    const bool pos = kk.x >= 0.f;
                    unsigned fl = 0;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const bool cert = fabsf(u[j]) > kk.w;
                        unc |= (unsigned)!cert << j;
                        fl |= (unsigned)(cert && ((u[j] >= 0.f) != pos)) << j;
                    }
                    fl &= vm;
                    if (__any_sync(0xffffffffu, fl)) {
                        if (fl) S.hit[at] = 1;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            if (!((fl >> j) & 1u)) continue;
                            // exactly one change in the layer below, none of its signs uncertain
                            if (((cprev >> (8 * j)) & 255u) == 1u && !((unc >> j) & 1u)) {
                                uint32_t* w = &S.prow[(iprev >> (8 * j)) & 255u][i >> 5];
                                const uint32_t b = 1u << (i & 31);
                                if (!(*reinterpret_cast<volatile uint32_t*>(w) & b)) atomicOr(w, b);
                            }
                            ccur += 1u << (8 * j);
                            icur = (icur & ~(255u << (8 * j))) | ((unsigned)(cb + i) & 127u) << (8 * j);
                        }
                    }
                }
            }
        }
    }
    // verdicts: undecided points go on, the others are final
    if (eq11) {
        neg = db & oa & ~(da | ob);
        und = ~(da | ob | neg);
    } else {
        und &= ~neg;  // one certainly negative difference decides
    }
    const unsigned bad = vm & (und | (cov ? unc : 0u)) & 15u;
    const unsigned adv = vm & neg & ~bad;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const unsigned long long t = tb + 32 * i + lane;
        const unsigned m = __ballot_sync(0xffffffffu, (adv >> i) & 1u);
        if (m) {
            acc.adv += (unsigned)__popc(m);
            const unsigned long long t0 = tb + 32 * i;
            const unsigned long long fi = t0 + (unsigned)(__ffs(m) - 1);
            acc.first = fi < acc.first ? fi : acc.first;
            if (lane == 0 && Q.bitmap && t0 < Q.bitmap_bits) atomicOr(&Q.bitmap[t0 >> 5], m);
        }
        queue_push_warp(out, (bad >> i) & 1u, t, q, Q.cnt, out_level);
    }
}

// The first pass over folded queries: groups of `group` tiles of mt points (mt a
// multiple of 32), claimed in order; a group's tiles may belong to several queries.
__global__ void __launch_bounds__(FT) k_fold(NetView net, const QueryView* __restrict__ qs, int nq,
                                             const unsigned long long* __restrict__ tile_prefix,
                                             unsigned long long ntiles, int mt, int group, int work_units,
                                             unsigned long long* claim, Queue out, int out_level) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FoldSm& S = *reinterpret_cast<FoldSm*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (nq == 1 && !folded(qs[0])) return;
    int cur = -1;
    bool small = true;
    for (int e = threadIdx.x; e < kFoldMax * kPairW; e += FT) (&S.prow[0][0])[e] = 0u;
    for (int e = threadIdx.x; e < kFoldMax + kFoldOut; e += FT) S.hit[e] = 0;
    // the sign changes and SS pairs of the query in work, into its masks
    auto flush = [&]() {
        const QueryView& Q = qs[cur];
        if (!Q.flip) return;
        const int L = net.L, nodes = S.f.nodes, offL = net.noff[L];
        for (int e = threadIdx.x; e < nodes + net.dims[L]; e += FT) {
            const int at = e < nodes ? e : kFoldMax + (e - nodes);
            if (!S.hit[at]) continue;
            S.hit[at] = 0;
            set_bit_once(Q.flip, (unsigned long long)(e < nodes ? Q.fnode[e] : offL + out_of_row(e - nodes, S.D)));
        }
        for (int e = threadIdx.x; e < nodes * kPairW; e += FT) {
            const int m = e / kPairW;
            uint32_t w = S.prow[m][e % kPairW];
            if (!w) continue;
            S.prow[m][e % kPairW] = 0u;
            int l = 1;
            while (m >= S.f.cb[l + 1] && l + 1 < L) ++l;  // node m's layer
            const int j = Q.fnode[m] - net.noff[l], Hn = net.dims[l + 1];
            while (w) {
                const int r = 32 * (e % kPairW) + __ffs(w) - 1;
                w &= w - 1u;
                const int i = l + 1 < L ? Q.fnode[S.f.cb[l + 1] + r] - net.noff[l + 1] : out_of_row(r, S.D);
                set_bit_once(Q.ss, (unsigned long long)net.ssoff[l] + (unsigned long long)j * Hn + i);
            }
        }
    };
    for (unsigned long long it = 0;; ++it) {
        if (threadIdx.x == 0)
            S.g = claim ? atomicAdd(claim, (unsigned long long)group)
                        : ((unsigned long long)blockIdx.x + it * gridDim.x) * group;
        __syncthreads();
        const unsigned long long ga = S.g;
        __syncthreads();  // every thread has read S.g before the next claim overwrites it
        if (ga >= ntiles) break;
        const unsigned long long gb = ga + group < ntiles ? ga + group : ntiles;
        int q = nq == 1 ? 0 : query_of_tile(tile_prefix, nq, ga);
        for (unsigned long long a = ga; a < gb; ++q) {
            const unsigned long long q0 = nq == 1 ? 0 : tile_prefix[q];
            const unsigned long long q1 = nq == 1 ? ntiles : tile_prefix[q + 1];
            const unsigned long long b = gb < q1 ? gb : q1;
            if (b <= a) continue;  // a query without tiles
            const QueryView& Q = qs[q];
            if (!folded(Q)) {
                a = b;
                continue;
            }
            if (q != cur) {
                if (cur >= 0) flush();
                __syncthreads();
                if (threadIdx.x == 0) {
                    fold_shape(net, Q, S.f);
                    S.D = Q.cnt->D;
                }
                for (int e = threadIdx.x; e < Q.s * Q.R; e += FT) S.xs[e] = Q.fxs[e];
                __syncthreads();
                small = S.f.entries <= kFoldSm;
                for (int e = threadIdx.x; small && e < S.f.entries; e += FT) {
                    const float4 c = Q.fc32[e];
                    S.co[2 * e] = make_float4(c.x, c.x, c.y, c.y);
                    S.co[2 * e + 1] = make_float4(c.z, c.z, c.w, c.w);
                }
                for (int e = threadIdx.x; e < S.f.nodes; e += FT) S.kc[e] = Q.fk32[e];
                for (int e = threadIdx.x; e < net.dims[net.L]; e += FT) S.kc[kFoldMax + e] = Q.fk32[kFoldMax + e];
                cur = q;
                __syncthreads();
            }
            const unsigned long long base = Q.lo & ~31ull;
            const unsigned long long ta = base + (a - q0) * (unsigned long long)mt;
            unsigned long long te = base + (b - q0) * (unsigned long long)mt;
            if (te > Q.hi) te = Q.hi;
            FoldAcc acc;
            for (unsigned long long tb = ta + (unsigned long long)(warp * FP); tb < te; tb += FW * FP) {
                if (small) fold_points<true>(net, Q, S, tb, te, acc, out, out_level, (unsigned)q);
                else fold_points<false>(net, Q, S, tb, te, acc, out, out_level, (unsigned)q);
            }
            if (lane == 0) {
                if (acc.adv) {
                    atomicAdd(&Q.cnt->n_adv, acc.adv);
                    atomicMin(&Q.cnt->first, acc.first);
                }
                if (acc.pts) atomicAdd(&Q.cnt->n_points, acc.pts);
            }
            __syncthreads();  // every push of the segment is out
            if (threadIdx.x == 0 && work_units) work_done(Q.cnt, b - a);
            a = b;
        }
    }
    if (cur >= 0) flush();
}

// ---- FP64 evaluation of one point by a warp

constexpr int F64W = 4;                  // warps per CTA of k_fold64
constexpr int kSetW = kFoldMax / 32 + 1;  // words of a set of nodes, then of outputs

struct Fold64 {
    double x[kMaxS + kFoldMax];        // the point's sources
    uint32_t ch[kSetW], ti[kSetW];     // rows that changed sign, rows whose sign is a tie
    int nch[kMaxL + 1], nti[kMaxL + 1];  // how many of each, per layer
};

// Point t of query Q by the definitions (Eq. 10 / Eq. 11 margin *m; signs and sign
// ties when coverage is on). A lane holds a row of a layer: its chain of FMAs over
// the sources is as long as the row, and a layer's rows run side by side (a few
// layers of at most a few dozen rows: a thread per point took 19 rows of 6..15
// columns one after the other). Returns false when some value lies within its
// error of the edge of the tie band, where FP64 rounding would decide.
__device__ bool fold64_point(const NetView& net, const QueryView& Q, Fold64& F, unsigned long long t, int lane,
                             double* m) {
    const int L = net.L, offL = net.noff[L], s = Q.s, D = Q.cnt->D;
    const bool cov = Q.flip != nullptr;
    __syncwarp();
    if (lane < kSetW) F.ch[lane] = F.ti[lane] = 0u;
    {
        int d[kMaxS];
        decode_digits(t, s, Q.R, d);
        for (int p = 0; p < s; ++p)
            if (lane == p) F.x[p] = (double)Q.dv[p * Q.R + d[p]] / 255.0;
    }
    bool edge = false;
    int cb = 0;
    double y = 0.0, ey = 0.0;
    for (int l = 1; l <= L; ++l) {
        const int nl = l < L ? Q.fst[2 + l] : net.dims[L], K = s + cb;
        int nch = 0, nti = 0;
        __syncwarp();  // the sources of the layers below are written
        for (int i0 = 0; i0 < nl; i0 += 32) {
            const int i = i0 + lane;
            bool ch = false, ti = false;
            if (i < nl) {
                const int nn = l < L ? Q.fnode[cb + i] : offL + out_of_row(i, D);
                const float2* row = Q.fco + (size_t)nn * Q.fstride;
                const double ub = Q.ub[nn], e = (double)Q.fe64[l < L ? cb + i : kFoldMax + i];
                double a = 0.0;
#pragma unroll 4
                for (int k = 0; k < K; ++k) {
                    const float2 c = row[k];
                    a = fma((double)c.x + (double)c.y, F.x[k], a);
                }
                const double u = ub + a;
                const bool base_tie = fabs(ub) < kTau;  // every evaluation of this neuron is a sign tie
                ti = fabs(u) < kTau || base_tie;
                ch = !ti && ((u >= 0.0) != (ub >= 0.0));
                edge = edge || (cov && !base_tie && fabs(fabs(u) - kTau) <= 2.0 * e);
                if (l < L) {
                    F.x[K + i] = fmax(u, 0.0) - fmax(ub, 0.0);
                } else {
                    y = u;
                    ey = e;
                }
                const int at = l < L ? cb + i : kFoldMax + i;
                if (ch) atomicOr(&F.ch[at >> 5], 1u << (at & 31));
                if (ti) atomicOr(&F.ti[at >> 5], 1u << (at & 31));
            }
            nch += __popc(__ballot_sync(0xffffffffu, ch));
            nti += __popc(__ballot_sync(0xffffffffu, ti));
        }
        if (lane == 0) {
            F.nch[l] = nch;
            F.nti[l] = nti;
        }
        if (l < L) cb += nl;
    }
    const int HL = net.dims[L];
    const double yD = __shfl_sync(0xffffffffu, y, 0);
    const double mx = warp_max(lane > 0 && lane < HL ? y : -DBL_MAX);
    const double em = warp_max(lane < HL ? ey : 0.0);
    *m = Q.prop == PROP_THRESHOLD ? fmax(yD - Q.V, Q.V - mx) : yD - mx;
    if (fabs(fabs(*m) - kTau) <= 4.0 * em + 0x1p-51 * (fabs(yD) + fabs(mx) + fabs(Q.V))) edge = true;
    __syncwarp();
    return !__any_sync(0xffffffffu, edge);
}

// Points k_fold left undecided.
__global__ void __launch_bounds__(32 * F64W) k_fold64(NetView net, const QueryView* __restrict__ qs,
                                                      const QEntry* __restrict__ in,
                                                      const unsigned long long* __restrict__ count,
                                                      unsigned long long cap, Queue out, int out_level) {
    __shared__ Fold64 Fs[F64W];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Fold64& F = Fs[warp];
    unsigned long long n = *count;
    if (n > cap) n = cap;
    const int L = net.L, offL = net.noff[L], HL = net.dims[L];
    for (unsigned long long e = (unsigned long long)blockIdx.x * F64W + warp; e < n;
         e += (unsigned long long)gridDim.x * F64W) {
        const QEntry en = in[e];
        const QueryView& Q = qs[en.q];
        if (!folded(Q)) continue;  // queued by another first pass
        const int D = Q.cnt->D;
        double m;
        if (!fold64_point(net, Q, F, en.t, lane, &m)) {
            if (lane == 0) {
                queue_push(out, en.t, en.q, Q.cnt, out_level);
                work_done(Q.cnt, 1);
            }
            continue;
        }
        if (lane == 0) {
            if (fabs(m) < kTau) {
                const unsigned long long k = atomicAdd(&Q.cnt->n_ties, 1ull);
                if (k < Q.ties_cap) Q.ties[k] = en.t;
                else atomicOr(&Q.cnt->err, DERR_TIES);
            } else if (m < 0.0) {
                record_adversarial(Q, en.t);
            }
        }
        if (Q.flip) {
            auto in_set = [](const uint32_t* w, int at) { return (w[at >> 5] >> (at & 31)) & 1u; };
            int c0 = 0;
            for (int l = 1; l <= L; ++l) {
                const int nl = l < L ? Q.fst[2 + l] : HL, b0 = l < L ? c0 : kFoldMax;
                const int b1 = l + 1 < L ? c0 + nl : kFoldMax;  // first row of the layer above
                const int nx = l + 1 < L ? Q.fst[3 + l] : HL;
                const int nch = F.nch[l], nti = F.nti[l];
                auto neuron = [&](int ll, int at, int i) { return ll < L ? Q.fnode[at + i] : offL + out_of_row(i, D); };
                for (int i = lane; i < nl; i += 32) {
                    const unsigned long long nn = (unsigned long long)neuron(l, b0, i);
                    if (in_set(F.ch, b0 + i)) set_bit_once(Q.flip, nn);
                    if (in_set(F.ti, b0 + i)) set_bit_once(Q.flip_tie, nn);
                }
                // SS pairs with layer l + 1: certain with one change and no tie in layer l;
                // under ties, the one change or (with none) each tie may be the only change
                if (l < L && (nti == 0 ? nch == 1 : nch <= 1)) {
                    for (int j = 0; j < nl; ++j) {
                        if (!in_set(nch == 1 ? F.ch : F.ti, b0 + j)) continue;
                        const unsigned long long r0 = (unsigned long long)net.ssoff[l] +
                            (unsigned long long)(Q.fnode[b0 + j] - net.noff[l]) * net.dims[l + 1];
                        for (int i = lane; i < nx; i += 32) {
                            const unsigned long long bit = r0 + (neuron(l + 1, b1, i) - net.noff[l + 1]);
                            if (nti == 0 && in_set(F.ch, b1 + i)) set_bit_once(Q.ss, bit);
                            else if (in_set(F.ch, b1 + i) || in_set(F.ti, b1 + i)) set_bit_once(Q.ss_tie, bit);
                        }
                    }
                }
                if (l < L) c0 += nl;
            }
        }
        __syncwarp();
        if (lane == 0) work_done(Q.cnt, 1);  // time to verdict: this point is resolved
    }
}

// FP64 margin of one point of query 0, where it folded (k_margin64 otherwise).
__global__ void __launch_bounds__(32) k_fold_margin(NetView net, const QueryView* __restrict__ qs,
                                                    unsigned long long t, double* out) {
    __shared__ Fold64 F;
    if (!folded(qs[0])) return;
    double m;
    fold64_point(net, qs[0], F, t, threadIdx.x, &m);
    if (threadIdx.x == 0) *out = m;
}

}  // namespace

bool fold_supported(const NetView& net) {
    return net.act == ACT_RELU && net.L >= 2 && net.dims[net.L] <= kFoldOut && net.hmax <= kMaxWidth;
}

size_t fold_coeff_entries(const NetView& net, int max_s) {
    // nodes in groups of 4 rows per layer, every row with at most max_s + kFoldMax columns
    return (size_t)(kFoldMax / 4 + net.L - 1 + (net.dims[net.L] + 3) / 4) * (max_s + kFoldMax);
}

void launch_fold_pack(const NetView& net, QueryView* d_qs, int nq, cudaStream_t st, unsigned long long* d_unfolded) {
    k_fold_pack<<<nq, 256, 0, st>>>(net, d_qs, d_unfolded);
}

void launch_fold(const NetView& net, const QueryView* d_qs, int nq, const unsigned long long* d_tile_prefix,
                 unsigned long long n_tiles, int mt, bool work_units, unsigned long long* claim, Queue out,
                 int out_level, int n_sm, cudaStream_t st) {
    cudaFuncSetAttribute(k_fold, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FoldSm));
    // a claim takes at least one round of the block's warps where the range has that many
    // points to hand out, and at most 16 rounds
    const unsigned long long per_round = (unsigned long long)(FT * 4 / mt), ctas = (unsigned long long)n_sm * 2;
    unsigned long long group = n_tiles / (ctas * 8);
    if (group > 16 * per_round) group = 16 * per_round;
    if (group >= per_round) group -= group % per_round;
    if (group < 1) group = 1;
    unsigned long long grid = (n_tiles + group - 1) / group;
    if (grid > ctas) grid = ctas;
    if (grid < 1) grid = 1;
    k_fold<<<(unsigned)grid, FT, sizeof(FoldSm), st>>>(net, d_qs, nq, d_tile_prefix, n_tiles, mt, (int)group,
                                                       work_units ? 1 : 0, claim, out, out_level);
}

void launch_fold64(const NetView& net, const QueryView* d_qs, const QEntry* in, const unsigned long long* count,
                   unsigned long long cap, Queue out, int out_level, int n_sm, cudaStream_t st) {
    k_fold64<<<(unsigned)n_sm * 4, 32 * F64W, 0, st>>>(net, d_qs, in, count, cap, out, out_level);
}

void launch_fold_margin(const NetView& net, const QueryView* d_qs, unsigned long long t, double* d_out,
                        cudaStream_t st) {
    k_fold_margin<<<1, 32, 0, st>>>(net, d_qs, t, d_out);
}

}  // namespace vbmc
