// fold.cu -- folded nets: the first pass over a ReLU net whose neurons mostly keep
// their sign in the box.
//
// Over one query's box (s pixels moved by at most k grey levels) a hidden neuron
// whose potential cannot cross zero acts linearly: its output change is its
// potential's change ("pos") or 0 ("neg"). The few others (the "nodes") act as their
// unperturbed sign says plus a correction where they cross: with u = ub + du,
//     relu(u) - relu(ub) = du + max(-u, 0)   (ub >= 0),   max(u, 0)   (ub < 0).
// Folding the linear parts into the weights leaves, exactly, a small net on the box:
//     du_n = sum_p A_np x_p + sum_m C_nm c_m,     x_p = dv_p / 255  (Eq. 1)
// over the s pixel changes and the corrections c_m >= 0 of the nodes of earlier
// layers, each 0 except at points where its node's sign has changed. Only nodes and
// outputs need evaluating: every other neuron's sign is known to be the unperturbed
// image's at every point, so it adds neither a sign change nor a sign tie (Sec. III-B).
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
// goes to the FP64 pass on the whole net. A query with more than kFoldMax nodes is not
// folded, nor one with a row, a base value or a bound that is not below kFoldBig (weights
// need only be finite, and rows are products of them); its general passes run instead
// (they return at once for folded queries). So every value here is finite.
//
// Error of k_fold, constant per row (a node, an output, a margin; u = 2^-24, K sources,
// M_n = |ub_n| + sum_k |c_nk| bound of source k): the FMA chain from the base value on
// and the roundings of c and x give at most (K + 8) u M_n, the sources' own errors sum |C_nm| e_m, the rows' fer_n, the
// base value |fl(ub) - ub| + eub. Their sum e_n
// bounds both |u_n - exact| and, since max(., 0) is 1-Lipschitz, |c_n - exact|.
// A sign is certain when |u_n|, a margin when its value exceeds e_n + 2 tau; one bound
// (the largest) serves all signs, one all margins that can come near 0.
//
// Why: on boxes of a few pixels moved by up to 15 grey levels about 1 % of the neurons
// can change sign, so a point costs a few hundred multiply-adds instead of the 268 k of
// 784-512-512-10 (or 2.1 M of 784-1024-1024-1024-10), in FP32 with a bound of about
// 1e-7 instead of a 16-bit screen's 1e-4..1e-2, and almost no point is left for a
// second pass. Whole calls, before and now: 784-512-512-10, s = 6, k = 7 (11.4 M
// points near the boundary) 38 -> 0.56 ms; 784-1024x3-10, s = 4, k = 15 with coverage
// 211 -> 0.64 ms (up to 0.99 where a point needs the FP64 pass); 784-300-100-10, s = 5,
// k = 9 in an L2 ball 27.5 -> 0.25 ms.
#include "counts.cuh"
#include "dev.cuh"
#include "dfloat.cuh"
#include "launch.h"

#include <algorithm>
#include <cfloat>

namespace vbmc {
namespace {

constexpr int FT = 256;          // threads of k_fold
constexpr int FW = FT / 32;
constexpr int FP = 4;            // points per thread: neighbours in the last pixel's digit
constexpr int kXp = 7;           // outer pixels whose changes a thread holds in registers
constexpr int kFoldSm = 1024;    // coefficient entries kept in shared memory (larger nets: through L1)
constexpr int kPairW = kFoldMax / 32;
// Steps of a thread (FP points each) between two additions of its 32-bit counts to the
// query's: one query's launch gives a warp its share of up to 2^62 points.
constexpr unsigned long long kFlushSteps = 1ull << 29;
static_assert(kFlushSteps * FP < (1ull << 32), "a thread's counts fit 32 bits between flushes");

// Rows and packed coefficients by layer: layer l's n[l] rows have s + cb[l] columns;
// the rows 4 g .. 4 g + 3 take 1 + s + cb[l] entries of fc32 from
// off[l] + g (1 + s + cb[l]) on: their base values, then column by column. Hidden
// layers: their nodes, each with the sign that makes its unperturbed potential
// negative. Output layer: for Eq. 10 the margins y_D - y_o (o != D, in order), filled
// up to a multiple of 4, then the outputs whose sign can change over the box (coverage
// on); for Eq. 11 every output.
struct FoldShape {
    int n[kMaxL + 1], cb[kMaxL + 1], off[kMaxL + 1];
    int entries, nodes, margins;  // margins: rows before the outputs (a multiple of 4)
};

__device__ void fold_shape(const NetView& net, const QueryView& Q, FoldShape& f) {
    int cb = 0, off = 0;
    for (int l = 1; l <= net.L; ++l) {
        const int n = Q.fst[2 + l];
        f.n[l] = n;
        f.cb[l] = cb;
        f.off[l] = off;
        off += ((n + 3) >> 2) * (1 + Q.s + cb);
        if (l < net.L) cb += n;
    }
    f.entries = off;
    f.nodes = cb;
    f.margins = Q.prop == PROP_THRESHOLD ? 0 : (net.dims[net.L] + 2) & ~3;
}

// Output i of the FP64 evaluation's order: D first, then the others in order.
__device__ __forceinline__ int out_of_row(int i, int D) { return i == 0 ? D : (i <= D ? i - 1 : i); }

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Base values of fill-up rows: a node that never crosses, a margin that never decides.
constexpr float kNoNode = -1.f, kNoMargin = 1e30f;

constexpr int kPackT = 512;

// Barrier of n threads of a block.
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

__global__ void __launch_bounds__(kPackT) k_fold_pack(NetView net, QueryView* qs, unsigned long long* unfolded) {
    __shared__ FoldShape f;
    __shared__ float eh[kFoldMax], eh64[kFoldMax], em_s[kPackT / 32], et_s[kPackT / 32];  // *_s: the warps' largest
    __shared__ int D_s, nv_s, big_s;
    __shared__ unsigned signs_s;
    chain_wait();
    chain_next();
    QueryView& Q = qs[blockIdx.x];
    if (!Q.fold || Q.fst[1] || (Q.cnt->err & DERR_PIXELS)) {
        if (threadIdx.x == 0 && unfolded) atomicAdd(unfolded, 1ull);
        return;
    }
    const int L = net.L, HL = net.dims[L], offL = net.noff[L], s = Q.s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool eq11 = Q.prop == PROP_THRESHOLD, cov = Q.flip != nullptr;
    if (threadIdx.x == 0) big_s = 0;
    __syncthreads();
    // rows' errors (FP32, rounded up): a warp per row, its lanes over the sources; layer
    // L + 1: the margins. Hidden rows depend on the layers below; outputs and margins on
    // all of them. The first half of the warps does the hidden layers while the other one
    // finds D and packs the coefficients: bound by the latency of dependent loads (one
    // after the other: D 3 us, coefficients 5, errors 6 on 784-512-512-10).
    const float tau2 = __double2float_ru(2.0 * kTau);
    float em = 0.f, et = 0.f;
    int D = 0;
    unsigned signs = 0;
    auto bound = [&](int l, int cb, int i) {
        const int n1 = l < L ? Q.fnode[cb + i] : (l == L ? offL + out_of_row(i, D) : offL + D);
        const int n2 = l <= L ? -1 : offL + (i < D ? i : i + 1);
        const float2* r1 = Q.fco + (size_t)n1 * Q.fstride;
        const float2* r2 = Q.fco + (size_t)(n2 < 0 ? n1 : n2) * Q.fstride;
        float M = 0.f, pr = 0.f, pr64 = 0.f;
        for (int k = lane; k < s + cb; k += 32) {
            float2 c = r1[k];
            if (n2 >= 0) c = df_add(c, make_float2(-r2[k].x, -r2[k].y));
            const float w = abs_up(c);
            if (k < s) {
                M = __fmaf_ru(w, Q.fx[k], M);
            } else {
                M = __fmaf_ru(w, __fadd_ru(Q.fsb[Q.fnode[k - s]], eh[k - s]), M);
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
        if (lane) return;
        double ub = Q.ub[n1];
        float fer = Q.fer[n1], eub = Q.fhe[n1].y;
        if (n2 >= 0) {
            ub -= Q.ub[n2];
            fer = __fadd_ru(fer, Q.fer[n2]);
            eub = __fadd_ru(eub, Q.fhe[n2].y);
        }
        const float ub32 = (float)ub;
        const float mag = __fadd_ru(__fadd_ru(fabsf(ub32), M), 1e-30f);
        float e = __fadd_ru(__fmaf_ru((float)(s + cb + 8) * 0x1p-24f, mag, pr), __fadd_ru(fer, 1e-37f));
        e = __fadd_ru(__fadd_ru(e, __double2float_ru(fabs((double)ub32 - ub))), eub);
        if (!(mag < kFoldBig) || !(e < kFoldBig)) big_s = 1;  // (or NaN)
        const float e2 = __fadd_ru(e, tau2);
        if (l > L) {
            // only a margin that can come near 0 over the box has a say in the common bound
            if (!(ub - (double)M - (double)e > 1e-3)) em = fmaxf(em, e2);
            return;
        }
        // the same in FP64 (u = 2^-53; x_p = dv_p / 255 rounds once, the rows' pairs are exact in it)
        const float e64 = __fmaf_ru((float)(s + cb + 12) * 0x1p-53f, mag, __fadd_ru(pr64, __fadd_ru(fer, eub)));
        Q.fe64[l < L ? cb + i : kFoldMax + i] = e64;
        const float thr = fabs(ub) < kTau ? INFINITY : e2;  // a base tie: every sign is a tie
        if (l < L) {
            eh[cb + i] = e;
            eh64[cb + i] = e64;
            et = fmaxf(et, thr);
        } else {
            const int o = out_of_row(i, D);
            Q.fk32[1 + o].y = e2;
            if ((signs >> o) & 1u) et = fmaxf(et, thr);
        }
    };
    if (warp < kPackT / 64) {
        int cb = 0;
        for (int l = 1; l < L; ++l) {
            const int rows = Q.fst[2 + l];
            for (int i = warp; i < rows; i += kPackT / 64) bound(l, cb, i);
            cb += rows;
            bar_sync(1, kPackT / 2);
        }
    } else {
        if (warp == kPackT / 64) {  // D: the largest output, the lowest index among equals; HL <= 32
            const double y = lane < HL ? Q.ub[offL + lane] : -DBL_MAX;
            const double top = warp_max(y);
            D = __ffs(__ballot_sync(0xffffffffu, lane < HL && y == top)) - 1;
            const double mx = warp_max(lane == D ? -DBL_MAX : y);
            // outputs that can change their sign over the box
            const bool cross = lane < HL && !(fabs(y) > ((double)Q.fbd[offL + lane] + (double)Q.fhe[offL + lane].y) *
                                                                (1.0 + 1e-6) + 4.0 * kTau);
            signs = __ballot_sync(0xffffffffu, cov && cross);
            if (lane == 0) {
                D_s = D;
                signs_s = signs;
                nv_s = eq11 ? HL : __popc(signs);  // rows that are outputs
                Q.cnt->D = D;
                Q.cnt->base_margin = eq11 ? fmax(top - Q.V, Q.V - mx) : top - mx;
                Q.fst[2 + L] = (eq11 ? 0 : (HL + 2) & ~3) + nv_s;
                fold_shape(net, Q, f);
            }
        }
        bar_sync(2, kPackT / 2);
        D = D_s;
        signs = signs_s;
        const int margins = f.margins;
        if (warp == kPackT / 64) {  // the outputs of the rows behind the margins; which of them have a sign test
            const bool row = lane < HL && (eq11 || ((signs >> lane) & 1u));
            const unsigned m = __ballot_sync(0xffffffffu, row);
            if (row) Q.forow[__popc(m & ((1u << lane) - 1u))] = lane | (int)((signs >> lane) & 1u) << 8;
        }
        bar_sync(2, kPackT / 2);
        // coefficient pair k of row i of layer l (k = -1: base value)
        auto coeff = [&](int l, int i, int k) -> float {
            if (l == L && i < margins) {
                const int o = i < D ? i : i + 1;
                if (o >= HL) return k < 0 ? kNoMargin : 0.f;
                if (k < 0) return (float)(Q.ub[offL + D] - Q.ub[offL + o]);
                const float2 a = Q.fco[(size_t)(offL + D) * Q.fstride + k], b = Q.fco[(size_t)(offL + o) * Q.fstride + k];
                return df_add(a, make_float2(-b.x, -b.y)).x;
            }
            if (i >= f.n[l]) return k < 0 ? kNoNode : 0.f;
            const int nn = l < L ? Q.fnode[f.cb[l] + i] : offL + (Q.forow[i - margins] & 255);
            const float c = k < 0 ? (float)Q.ub[nn] : Q.fco[(size_t)nn * Q.fstride + k].x;
            return l < L && Q.fcls[nn] == 3 ? -c : c;
        };
        for (int e = threadIdx.x - kPackT / 2; e < f.entries; e += kPackT / 2) {
            int l = L;
            while (e < f.off[l]) --l;  // layers without rows have the offset of the next one
            const int cols = 1 + s + f.cb[l], g = (e - f.off[l]) / cols, k = e - f.off[l] - g * cols - 1;
            Q.fc32[e] = make_float4(coeff(l, 4 * g, k), coeff(l, 4 * g + 1, k), coeff(l, 4 * g + 2, k),
                                    coeff(l, 4 * g + 3, k));
        }
    }
    __syncthreads();
    D = D_s;
    signs = signs_s;
    for (int i = warp; i < HL + (eq11 ? 0 : HL - 1); i += kPackT / 32) {
        if (i < HL) bound(L, f.nodes, i);
        else bound(L + 1, f.nodes, i - HL);
    }
    if (lane == 0) {
        em_s[warp] = em;
        et_s[warp] = et;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kPackT / 32; ++w) {
            em = fmaxf(em, em_s[w]);
            et = fmaxf(et, et_s[w]);
        }
        if (big_s) {
            Q.fst[1] = 1;
            if (unfolded) atomicAdd(unfolded, 1ull);
            return;
        }
        Q.fk32[0] = make_float4(em, et, 0.f, 0.f);
        Q.fst[0] = 1;
        Q.cnt->folded = 1;
    }
}

struct FoldSm {
    float4 co[kFoldSm];                  // fc32
    float ey[kFoldOut];                  // Eq. 11: error bounds of the outputs
    int orow[kFoldOut];                  // forow
    float em, thr;                       // what every margin, every sign has to exceed
    float xs[kMaxS * kMaxR];             // [s][R] fl(dv / 255)
    uint32_t prow[kFoldMax][kPairW];     // SS pairs of node m with row i of the next layer
    uint4 fl[FW][kFoldMax];              // per warp: the points at which a node's sign has changed
    unsigned char hit[kFoldMax + kFoldOut];  // nodes and outputs that changed sign at some point
    FoldShape f;
    int D;
    unsigned long long g;
};

// x / d and the remainder by the 32-bit reciprocal inv = floor((2^32 - 1) / d): the
// product's high word is at most one too small.
__device__ __forceinline__ unsigned divmod(unsigned x, unsigned d, unsigned inv, unsigned& r) {
    unsigned q = __umulhi(x, inv);
    r = x - q * d;
    if (r >= d) {
        r -= d;
        ++q;
    }
    return q;
}

// The range [ta, te) of a query as units: the 4-digit pieces of the last pixel's digit
// behind each prefix (the digits of the others), numbered in order of their points.
struct FoldUnits {
    unsigned long long pa, n;  // first prefix, number of units
    unsigned Rl, C, cinv, ca;  // last digit's range, pieces per prefix, 1 / C, first piece
    bool pf32;                 // prefixes fit 32 bits
    __device__ FoldUnits(const QueryView& Q, unsigned long long ta, unsigned long long te) {
        Rl = Q.s > 0 ? (unsigned)Q.R : 1u;
        C = (Rl + FP - 1) / FP;
        cinv = 0xFFFFFFFFu / C;
        pa = ta / Rl;
        const unsigned long long pe = (te - 1) / Rl;
        ca = (unsigned)(ta - pa * Rl) / FP;
        n = (pe - pa) * C + (unsigned)(te - 1 - pe * Rl) / FP - ca + 1;
        pf32 = pe <= 0xFFFFFFFFull;
    }
    __device__ unsigned long long prefix(unsigned long long u, unsigned& c) const {
        const unsigned long long x = ca + u;
        if (x <= 0xFFFFFFFFull) return pa + divmod((unsigned)x, C, cinv, c);
        c = (unsigned)(x % C);
        return pa + x / C;
    }
};

// FP points of query Q: digits 4 c .. 4 c + 3 of the last pixel behind prefix pf, those
// of [ta, te). Every lane of the warp calls it, on units that are consecutive over the
// lanes (so are the points); on: the lane has one. Loops that few points need (64-bit
// prefixes, filters, sign changes) stay rolled: unrolled, the body outgrew the
// instruction cache (2.1 of 8 stalls per instruction).
template <bool SM>
__device__ __forceinline__ void fold_points(const NetView& net, const QueryView& Q, FoldSm& S,
                                            unsigned long long pf, unsigned c, bool on, bool pf32,
                                            unsigned long long ta, unsigned long long te, PointCounts& acc,
                                            const Queue& out, int out_level, unsigned q) {
    const int lane = threadIdx.x & 31;
    const int s = Q.s, R = Q.R, L = net.L;
    const int np = s > 0 ? s - 1 : 0, sl = s - np, Rl = s > 0 ? R : 1;
    const bool cov = Q.flip != nullptr;
    float4 src[kFoldMax];           // sources of the nodes that some lane of the warp has crossed
    const unsigned long long t0 = pf * (unsigned)Rl + 4 * c;
    unsigned vm = 0;                // bit j: point t0 + j is checked
#pragma unroll
    for (int j = 0; j < FP; ++j)
        vm |= (unsigned)(on && (int)(4 * c) + j < Rl && t0 + j >= ta && t0 + j < te) << j;
    float xp[kXp], xl[FP] = {0.f, 0.f, 0.f, 0.f};  // changes of the first outer pixels, of the last one
    unsigned long long dlo = 0, dhi = 0;  // with more of them: the digits, a byte each, pixel 0 lowest
    auto digit = [&](int p) { return (int)((p < 8 ? dlo >> (8 * p) : dhi >> (8 * (p - 8))) & 255u); };
    const bool filt = Q.filter != 0;
    int l2 = 0;                     // the filter: squared changes (fl(dv / 255) times 255 is within 1e-4 of dv)
    bool shell = Q.k == 0;
    auto test = [&](float x, int d) {
        const int v = __float2int_rn(x * 255.f);
        l2 += v * v;
        shell = shell || d == 0 || d == R - 1;
    };
    {
        const unsigned inv = 0xFFFFFFFFu / (unsigned)R;
        if (pf32 && np <= kXp) {
            unsigned x = (unsigned)pf, d;
#pragma unroll
            for (int p = kXp - 1; p >= 0; --p) {
                if (p >= np) continue;
                x = divmod(x, (unsigned)R, inv, d);
                xp[p] = S.xs[p * R + (int)d];
                if (filt) test(xp[p], (int)d);
            }
        } else {
            unsigned long long x = pf;
#pragma unroll 1
            for (int p = np - 1; p >= 0; --p) {
                const unsigned d = (unsigned)(x % (unsigned)R);
                x /= (unsigned)R;
                dhi = (dhi << 8) | (dlo >> 56);
                dlo = (dlo << 8) | d;
                if (filt) test(S.xs[p * R + (int)d], (int)d);
            }
#pragma unroll
            for (int p = 0; p < kXp; ++p)
                if (p < np) xp[p] = S.xs[p * R + digit(p)];
        }
    }
    if (sl) {
#pragma unroll
        for (int j = 0; j < FP; ++j) xl[j] = S.xs[np * R + min((int)(4 * c) + j, R - 1)];
    }
    if (filt) {
#pragma unroll
        for (int j = 0; j < FP; ++j) {
            const int d = (int)(4 * c) + j, v = __float2int_rn(xl[j] * 255.f);
            const bool on_shell = shell || (sl && (d == 0 || d == R - 1));
            if (((Q.filter & FILTER_L2) && (long long)(l2 + v * v) > Q.l2max) ||
                ((Q.filter & FILTER_SHELL) && !on_shell))
                vm &= ~(1u << j);
        }
        acc.pts += __popc(vm);
    }
    unsigned act[kFoldMax / 32] = {};  // nodes with a source that is not 0 at all the warp's points
    float least[FP], mn[FP];  // least |u| over the signs near 0 or changed; least margin
#pragma unroll
    for (int j = 0; j < FP; ++j) least[j] = mn[j] = INFINITY;
    const float thr = S.thr;  // every sign is certain beyond it
    unsigned da = 0, db = 0, oa = 0, ob = 15u;  // Eq. 11: sides of V
    const bool eq11 = Q.prop == PROP_THRESHOLD;
    // sign changes as sets of the warp's 128 points (word j: point j of every lane): of the
    // layer in work the points with a change and with two, of the layer below those with
    // exactly one and no uncertain sign so far
    unsigned VM[FP], c1[FP], c2[FP], ex[FP] = {0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < FP; ++j) VM[j] = __ballot_sync(0xffffffffu, (vm >> j) & 1u);
    int cbp = 0;  // first node of the layer below
    // row i of the layer has changed its sign for certain at the points F
    auto changed = [&](const unsigned (&F)[FP], int i, int at, int cb) {
        if (!(F[0] | F[1] | F[2] | F[3])) return;
        S.hit[at] = 1;
        if ((ex[0] | ex[1] | ex[2] | ex[3])) {  // SS: the node m of the layer below is its only change
            for (int m = cbp + lane; m < cb; m += 32) {
                const unsigned aw = m < 64 ? (m < 32 ? act[0] : act[1]) : (m < 96 ? act[2] : act[3]);
                if (!((aw >> (m & 31)) & 1u)) continue;
                const uint4 G = S.fl[threadIdx.x >> 5][m];
                if ((G.x & ex[0] & F[0]) | (G.y & ex[1] & F[1]) | (G.z & ex[2] & F[2]) | (G.w & ex[3] & F[3])) {
                    const uint32_t b = 1u << (i & 31);
                    uint32_t* w = &S.prow[m][i >> 5];
                    if (!(*reinterpret_cast<volatile uint32_t*>(w) & b)) atomicOr(w, b);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < FP; ++j) {
            c2[j] |= c1[j] & F[j];
            c1[j] |= F[j];
        }
    };
#pragma unroll 1
    for (int l = 1; l <= L; ++l) {
        const int n = S.f.n[l], cb = S.f.cb[l], cols = 1 + s + cb;
#pragma unroll
        for (int j = 0; j < FP; ++j) c1[j] = c2[j] = 0u;
        const float4* co = (SM ? S.co : Q.fc32) + S.f.off[l];
#pragma unroll 1
        for (int i0 = 0; i0 < n; i0 += 4, co += cols) {
            float4 b = co[0];  // the base values and the outer pixels' part, the same at the 4 points
#pragma unroll
            for (int p = 0; p < kXp; ++p) {
                if (p >= np) break;
                const float4 w = co[1 + p];
                b.x = fmaf(w.x, xp[p], b.x);
                b.y = fmaf(w.y, xp[p], b.y);
                b.z = fmaf(w.z, xp[p], b.z);
                b.w = fmaf(w.w, xp[p], b.w);
            }
#pragma unroll 1
            for (int p = kXp; p < np; ++p) {
                const float4 w = co[1 + p];
                const float x = S.xs[p * R + digit(p)];
                b.x = fmaf(w.x, x, b.x);
                b.y = fmaf(w.y, x, b.y);
                b.z = fmaf(w.z, x, b.z);
                b.w = fmaf(w.w, x, b.w);
            }
            float a[4][FP];
            {
                const float4 w = sl ? co[1 + np] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int j = 0; j < FP; ++j) {
                    a[0][j] = fmaf(w.x, xl[j], b.x);
                    a[1][j] = fmaf(w.y, xl[j], b.y);
                    a[2][j] = fmaf(w.z, xl[j], b.z);
                    a[3][j] = fmaf(w.w, xl[j], b.w);
                }
            }
#pragma unroll
            for (int w = 0; w < kFoldMax / 32; ++w) {
                const int own = cb - 32 * w;  // this layer's own nodes are no sources
                if (own <= 0) break;
#pragma unroll 1
                for (unsigned m = own >= 32 ? act[w] : act[w] & ((1u << own) - 1u); m; m &= m - 1u) {
                    const int k = 32 * w + __ffs(m) - 1;
                    const float4 v4 = src[k], c4 = co[1 + s + k];
                    const float v[FP] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
                    for (int j = 0; j < FP; ++j) {
                        a[0][j] = fmaf(c4.x, v[j], a[0][j]);
                        a[1][j] = fmaf(c4.y, v[j], a[1][j]);
                        a[2][j] = fmaf(c4.z, v[j], a[2][j]);
                        a[3][j] = fmaf(c4.w, v[j], a[3][j]);
                    }
                }
            }
            if (l < L) {  // potentials with the sign that makes the unperturbed ones negative
                float top[4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    top[e] = fmaxf(fmaxf(a[e][0], a[e][1]), fmaxf(a[e][2], a[e][3]));
                // below -thr everywhere: no change, nothing uncertain, no source
                if (!__any_sync(0xffffffffu, fmaxf(fmaxf(top[0], top[1]), fmaxf(top[2], top[3])) >= -thr)) continue;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (i0 + e >= n || !__any_sync(0xffffffffu, top[e] >= -thr)) continue;
                    const int at = cb + i0 + e;
                    src[at] = make_float4(fmaxf(a[e][0], 0.f), fmaxf(a[e][1], 0.f), fmaxf(a[e][2], 0.f),
                                          fmaxf(a[e][3], 0.f));
#pragma unroll
                    for (int w = 0; w < kFoldMax / 32; ++w) act[w] |= (at >> 5) == w ? 1u << (at & 31) : 0u;
                    if (cov) {
                        unsigned F[FP];
#pragma unroll
                        for (int j = 0; j < FP; ++j) {
                            least[j] = fminf(least[j], fabsf(a[e][j]));
                            F[j] = __ballot_sync(0xffffffffu, a[e][j] > thr) & VM[j];
                        }
                        if (lane == 0) S.fl[threadIdx.x >> 5][at] = make_uint4(F[0], F[1], F[2], F[3]);
                        changed(F, i0 + e, at, cb);
                    }
                }
                continue;
            }
            if (i0 < S.f.margins) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
#pragma unroll
                    for (int j = 0; j < FP; ++j) mn[j] = fminf(mn[j], a[e][j]);
                }
                continue;
            }
#pragma unroll 1
            for (int e = 0; e < 4 && i0 + e < n; ++e) {  // outputs: their signs, Eq. 11
                float y[FP];
#pragma unroll
                for (int j = 0; j < FP; ++j) y[j] = e < 2 ? (e ? a[1][j] : a[0][j]) : (e < 3 ? a[2][j] : a[3][j]);
                const int w = S.orow[i0 + e - S.f.margins], o = w & 255;
                const float base = e < 2 ? (e ? co[0].y : co[0].x) : (e < 3 ? co[0].z : co[0].w);
                if (eq11) {
#pragma unroll
                    for (int j = 0; j < FP; ++j) {
                        const int sd = thr_side(y[j], (float)Q.V, S.ey[o]);
                        if (o == S.D) {
                            da |= (unsigned)(sd > 0) << j;
                            db |= (unsigned)(sd < 0) << j;
                        } else {
                            oa |= (unsigned)(sd > 0) << j;
                            if (!(sd < 0)) ob &= ~(1u << j);
                        }
                    }
                }
                if (w >> 8) {
                    unsigned F[FP];
#pragma unroll
                    for (int j = 0; j < FP; ++j) {
                        least[j] = fminf(least[j], fabsf(y[j]));
                        F[j] = VM[j] & __ballot_sync(0xffffffffu, fabsf(y[j]) > thr && ((y[j] >= 0.f) != (base >= 0.f)));
                    }
                    changed(F, o, kFoldMax + o, cb);
                }
            }
        }
        if (cov) {
#pragma unroll
            for (int j = 0; j < FP; ++j) ex[j] = c1[j] & ~c2[j];
            if (ex[0] | ex[1] | ex[2] | ex[3]) {
#pragma unroll
                for (int j = 0; j < FP; ++j) ex[j] &= __ballot_sync(0xffffffffu, least[j] > thr);
                __syncwarp();  // the layer's sets of points are written
            }
        }
        cbp = cb;
    }
    // verdicts: undecided points go on, the others are final
    unsigned neg = 0, und = 0, unc = 0;
    if (eq11) {
        neg = db & oa & ~(da | ob);
        und = ~(da | ob | neg);
    } else {
        const float em = S.em;
#pragma unroll
        for (int j = 0; j < FP; ++j) {
            neg |= (unsigned)(mn[j] < -em) << j;
            und |= (unsigned)!(fabsf(mn[j]) > em) << j;
        }
    }
    if (cov) {
#pragma unroll
        for (int j = 0; j < FP; ++j) unc |= (unsigned)!(least[j] > thr) << j;
    }
    const unsigned bad = vm & (und | unc) & 15u;
    const unsigned adv = vm & neg & ~bad;
    if (__any_sync(0xffffffffu, adv)) {
        if (adv) {
            acc.adv += __popc(adv);
            const unsigned long long f = t0 + (unsigned)(__ffs(adv) - 1);
            acc.first = f < acc.first ? f : acc.first;
        }
        if (Q.bitmap) {  // the warp's points are consecutive: at most 128, in 5 words
            const unsigned long long w0 = __shfl_sync(0xffffffffu, t0, 0) >> 5;
            const unsigned at = (unsigned)(t0 - (w0 << 5)), wi = at >> 5, sh = at & 31u;
#pragma unroll
            for (unsigned w = 0; w < 5; ++w) {
                const unsigned part = wi == w ? adv << sh : (sh > 28u && wi + 1 == w ? adv >> (32u - sh) : 0u);
                const unsigned m = __reduce_or_sync(0xffffffffu, part);
                if (m && lane == 0 && ((w0 + w) << 5) < Q.bitmap_bits) atomicOr(&Q.bitmap[w0 + w], m);
            }
        }
    }
    if (__any_sync(0xffffffffu, bad)) {
#pragma unroll 1
        for (int j = 0; j < FP; ++j) queue_push_warp(out, (bad >> j) & 1u, t0 + j, q, Q.cnt, out_level);
    }
}

// The first pass over folded queries. One query: its units lie in rounds over all the
// launch's warps. Many: groups of `group` tiles of mt points (mt a multiple of 32),
// claimed in order; a group's tiles may belong to several queries.
// A thread takes 4 points that differ in the last pixel's digit only: they share the
// decode and the outer pixels' part of every row, and a row's coefficients, read as
// shared-memory broadcasts, serve 4 points. A node's source is 0 until its sign
// changes, so a warp adds up only those that one of its 128 points has crossed, and
// looks at a node's sign only where the largest of its potentials comes near 0 (one
// vote for 4 nodes). Sign changes are sets of points in 4 words, the same in every
// lane. Bound by issue slots (2.3 a cycle at 16 warps per SM; 3 CTAs per SM spill and
// are slower: 200 -> 215 us). Before (every source added, a point per register set and
// its outer pixels' part each, signs point by point) and now: 784-512-512-10, s = 6,
// k = 7 (11.4 M points) 356 -> 199 us, 784-1024x3-10, s = 4, k = 15 337 -> 97 us, the
// last wave of 64 queries on 784-256-256-10 1,255 -> 665 us.
__global__ void __launch_bounds__(FT, 2) k_fold(NetView net, const QueryView* __restrict__ qs, int nq,
                                                unsigned long long lo, unsigned long long hi,
                                                const unsigned long long* __restrict__ tile_prefix,
                                                unsigned long long ntiles, int mt, int group, int work_units,
                                                unsigned long long* claim, Queue out, int out_level) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FoldSm& S = *reinterpret_cast<FoldSm*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    chain_wait();  // (no chain_next: waiting blocks of k_fold64 take shared memory from this kernel's L1)
    if (nq == 1 && !folded(qs[0])) return;
    int cur = -1;
    bool small = true;
    for (int e = threadIdx.x; e < kFoldMax * kPairW; e += FT) (&S.prow[0][0])[e] = 0u;
    for (int e = threadIdx.x; e < kFoldMax + kFoldOut; e += FT) S.hit[e] = 0;
    auto load = [&](int q) {  // query q's coefficients and constants
        const QueryView& Q = qs[q];
        if (threadIdx.x == 0) {
            fold_shape(net, Q, S.f);
            S.D = Q.cnt->D;
            S.em = Q.fk32[0].x;
            S.thr = Q.fk32[0].y;
        }
        for (int e = threadIdx.x; e < Q.s * Q.R; e += FT) S.xs[e] = Q.fxs[e];
        if (threadIdx.x < net.dims[net.L]) {
            S.ey[threadIdx.x] = Q.fk32[1 + threadIdx.x].y;
            S.orow[threadIdx.x] = Q.forow[threadIdx.x];
        }
        __syncthreads();
        small = S.f.entries <= kFoldSm;
        for (int e = threadIdx.x; small && e < S.f.entries; e += FT) S.co[e] = Q.fc32[e];
        cur = q;
        __syncthreads();
    };
    // the sign changes and SS pairs of the query in work, into its masks
    auto flush = [&]() {
        const QueryView& Q = qs[cur];
        if (!Q.flip) return;
        const int L = net.L, nodes = S.f.nodes, offL = net.noff[L];
        for (int e = threadIdx.x; e < nodes + net.dims[L]; e += FT) {
            const int at = e < nodes ? e : kFoldMax + (e - nodes);
            if (!S.hit[at]) continue;
            S.hit[at] = 0;
            set_bit_once(Q.flip, (unsigned long long)(e < nodes ? Q.fnode[e] : offL + (e - nodes)));
        }
        for (int e = threadIdx.x; e < nodes * kPairW; e += FT) {
            const int m = e / kPairW;
            uint32_t w = S.prow[m][e % kPairW];
            if (!w) continue;
            S.prow[m][e % kPairW] = 0u;
            int l = 1;
            while (l + 1 < L && m >= S.f.cb[l + 1]) ++l;  // node m's layer
            const int j = Q.fnode[m] - net.noff[l], Hn = net.dims[l + 1];
            while (w) {
                const int r = 32 * (e % kPairW) + __ffs(w) - 1;
                w &= w - 1u;
                const int i = l + 1 < L ? Q.fnode[S.f.cb[l + 1] + r] - net.noff[l + 1] : r;
                set_bit_once(Q.ss, (unsigned long long)net.ssoff[l] + (unsigned long long)j * Hn + i);
            }
        }
    };
    // units u0 + stride i of [ta, te), 32 per warp and step, then the warp's counts
    auto segment = [&](int q, unsigned long long ta, unsigned long long te, unsigned long long u0,
                       unsigned long long stride) {
        const QueryView& Q = qs[q];
        PointCounts acc;
        if (ta < te) {
            const FoldUnits U(Q, ta, te);
            for (unsigned long long u = u0; u < U.n;) {
                const unsigned long long end = U.n - u > stride * kFlushSteps ? u + stride * kFlushSteps : U.n;
                for (; u < end; u += stride) {
                    unsigned c;
                    const unsigned long long pf = U.prefix(u + lane, c);
                    const bool on = u + lane < U.n;
                    if (small) fold_points<true>(net, Q, S, pf, c, on, U.pf32, ta, te, acc, out, out_level, (unsigned)q);
                    else fold_points<false>(net, Q, S, pf, c, on, U.pf32, ta, te, acc, out, out_level, (unsigned)q);
                }
                acc.flush(Q.cnt);
            }
        }
        __syncthreads();  // every push of the segment is out
    };
    if (nq == 1) {
        load(0);
        // consecutive pieces go to different CTAs, so that a small range spreads
        segment(0, lo, hi, 32ull * (blockIdx.x + gridDim.x * (unsigned)warp), 32ull * gridDim.x * FW);
        flush();
        __syncthreads();
        if (threadIdx.x == 0 && work_units)  // the launch's share of the query's tiles
            work_done(qs[0].cnt, ntiles * (blockIdx.x + 1ull) / gridDim.x - ntiles * blockIdx.x / gridDim.x);
        return;
    }
    for (;;) {
        if (threadIdx.x == 0) S.g = atomicAdd(claim, (unsigned long long)group);
        __syncthreads();
        const unsigned long long ga = S.g;
        __syncthreads();  // every thread has read S.g before the next claim overwrites it
        if (ga >= ntiles) break;
        const unsigned long long gb = ga + group < ntiles ? ga + group : ntiles;
        int q = query_of_tile(tile_prefix, nq, ga);
        for (unsigned long long a = ga; a < gb; ++q) {
            const unsigned long long q0 = tile_prefix[q], q1 = tile_prefix[q + 1];
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
                load(q);
            }
            const unsigned long long base = Q.lo & ~31ull;
            const unsigned long long ta = base + (a - q0) * (unsigned long long)mt;
            const unsigned long long te = base + (b - q0) * (unsigned long long)mt;
            segment(q, ta < Q.lo ? Q.lo : ta, te > Q.hi ? Q.hi : te, 32ull * warp, 32ull * FW);
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
                edge = edge || (cov && !base_tie && !(fabs(fabs(u) - kTau) > 2.0 * e));
                if (l < L) {
                    F.x[K + i] = fmax(ub >= 0.0 ? -u : u, 0.0);
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
    if (!(fabs(fabs(*m) - kTau) > 4.0 * em + 0x1p-51 * (fabs(yD) + fabs(mx) + fabs(Q.V)))) edge = true;
    __syncwarp();
    return !__any_sync(0xffffffffu, edge);
}

// Points k_fold left undecided.
__global__ void __launch_bounds__(32 * F64W) k_fold64(NetView net, const QueryView* __restrict__ qs,
                                                      const QEntry* in, const unsigned long long* count,
                                                      unsigned long long cap, Queue out, int out_level) {
    __shared__ Fold64 Fs[F64W];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Fold64& F = Fs[warp];
    chain_wait();
    chain_next();
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

}  // namespace

bool fold_supported(const NetView& net) {
    return net.act == ACT_RELU && net.L >= 2 && net.dims[net.L] <= kFoldOut && net.hmax <= kMaxWidth;
}

size_t fold_coeff_entries(const NetView& net, int max_s) {
    // nodes in groups of 4 rows per layer, every row with at most 1 + max_s + kFoldMax entries
    return (size_t)(kFoldMax / 4 + net.L - 1 + (net.dims[net.L] + 2) / 4 + (net.dims[net.L] + 3) / 4) *
           (1 + max_s + kFoldMax);
}

void launch_fold_pack(const NetView& net, QueryView* d_qs, int nq, cudaStream_t st, unsigned long long* d_unfolded) {
    launch_chained(k_fold_pack, nq, kPackT, 0, st, net, d_qs, d_unfolded);
}

void launch_fold(const NetView& net, const QueryView* d_qs, int nq, unsigned long long lo, unsigned long long hi,
                 const unsigned long long* d_tile_prefix, unsigned long long n_tiles, int mt, bool work_units,
                 unsigned long long* claim, Queue out, int out_level, int n_sm, cudaStream_t st) {
    cudaFuncSetAttribute(k_fold, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FoldSm));
    const unsigned long long ctas = (unsigned long long)n_sm * 2;
    // one query: a warp for every 32 units of up to 4 points, as many as fit. Many: a claim
    // takes 16 rounds of the block's warps, fewer where the CTAs would not get 2 claims each
    const unsigned long long per_round = (unsigned long long)(FT * FP / mt);
    unsigned long long group = std::min<unsigned long long>(n_tiles / (ctas * 2), 16 * per_round);
    if (group < 1) group = 1;
    unsigned long long grid = nq == 1 ? (hi - lo + 127) / 96 : (n_tiles + group - 1) / group;
    if (grid > ctas) grid = ctas;
    if (grid < 1) grid = 1;
    launch_chained(k_fold, (unsigned)grid, FT, sizeof(FoldSm), st, net, d_qs, nq, lo, hi, d_tile_prefix, n_tiles, mt,
                   (int)group, work_units ? 1 : 0, claim, out, out_level);
}

void launch_fold64(const NetView& net, const QueryView* d_qs, const QEntry* in, const unsigned long long* count,
                   unsigned long long cap, Queue out, int out_level, int n_sm, cudaStream_t st) {
    launch_chained(k_fold64, (unsigned)n_sm * 4, 32 * F64W, 0, st, net, d_qs, in, count, cap, out, out_level);
}

}  // namespace vbmc
