// prologue.cu -- per-query set-up that every pass over the points uses.
//
//  * k_pro_init:   validate the pixel list, build the clipped step table
//                  dv[p][d] = clamp(v_p + d - k, 0, 255) - v_p, reset counters
//  * k_pro_layer:  FP64 activation potentials of the unperturbed image, one
//                  layer per launch (Eq. 1; Eq. 2 or ReLU on hidden layers)
//  * k_pro_tables: layer-1 delta tables tab[p][d][j] = W_1[j][p] * dv[p][d] / 255,
//                  so a point's layer-1 potential is ub_1 + sum_p tab[p][d_p]
//                  (the incremental first layer: s table adds instead of an
//                  H_0-long dot product per neuron)
//  * k_pro_finish: class D and margin of the unperturbed image, and the
//                  per-neuron constants of the screens' error bounds
#include "dev.cuh"
#include "dfloat.cuh"
#include "launch.h"

#include <cfloat>

namespace vbmc {

__global__ void k_pro_init(NetView net, QueryView* qs, int nq) {
    if (blockIdx.x == 0) {  // W_1 comes in meanwhile
        const size_t n1 = (size_t)net.dims[0] * net.dims[1];
        for (size_t j = 32 * ((size_t)blockIdx.y * blockDim.x + threadIdx.x); j < n1; j += 32 * (size_t)gridDim.y * blockDim.x)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(net.W[1] + j));
    }
    chain_wait();
    chain_next();
    QueryView& Q = qs[blockIdx.x];
    const int H0 = net.dims[0];
    if (blockIdx.y == 0 && threadIdx.x < 32) {
        const int p = threadIdx.x;
        const bool own = Q.s >= 0 && Q.s <= kMaxS && p < Q.s;
        const int v = own ? Q.pix_in[p] : -1 - p;
        const unsigned same = __match_any_sync(0xffffffffu, v);
        // in range, and in no other lane
        const bool bad = own && (v < 0 || v >= H0 || __popc(same) > 1);
        const bool ok = Q.s >= 0 && Q.s <= kMaxS && !__any_sync(0xffffffffu, bad);
        if (own) Q.pix[p] = (ok && v >= 0 && v < H0) ? v : 0;  // never index out of range
        if (p == 0) {
            Counters* c = Q.cnt;
            c->n_adv = 0;
            c->first = ~0ull;
            c->n_ties = 0;
            c->n_q[0] = c->n_q[1] = c->n_q[2] = c->n_q[3] = 0;
            c->n_points = Q.filter ? 0ull : Q.hi - Q.lo;  // with a filter the passes count
            c->err = ok ? 0u : DERR_PIXELS;
            c->D = 0;
            c->base_margin = 0.0;
            c->t0 = globaltimer_ns();
            c->t_final = 0;
            c->work = Q.ntiles;
            c->folded = 0;
            if (Q.fst) Q.fst[0] = Q.fst[1] = 0;
        }
    }
    if (Q.image_keep && blockIdx.y == 0)
        for (int j = threadIdx.x; j < H0; j += blockDim.x) Q.image_keep[j] = Q.image[j];
    // results start from zero on every call
    const int nb = gridDim.y, bt = blockIdx.y * blockDim.x + threadIdx.x, nt = nb * blockDim.x;
    if (Q.flip)
        for (int w = bt; w < net.flip_words; w += nt) Q.flip[w] = Q.flip_tie[w] = 0u;
    if (Q.ss)
        for (int w = bt; w < net.ss_words; w += nt) Q.ss[w] = Q.ss_tie[w] = 0u;
    if (Q.bitmap && Q.hi > 0) {
        const unsigned long long nw = (Q.hi + 31) / 32;
        uint4* b4 = reinterpret_cast<uint4*>(Q.bitmap);
        for (unsigned long long w = bt; w < nw / 4; w += nt) b4[w] = make_uint4(0, 0, 0, 0);
        for (unsigned long long w = (nw / 4) * 4 + bt; w < nw; w += nt) Q.bitmap[w] = 0u;
    }
    if (blockIdx.y != 0) return;
    __syncthreads();
    for (int e = threadIdx.x; e < Q.s * Q.R; e += blockDim.x) {
        int p = e / Q.R, d = e % Q.R;
        int v = Q.image[Q.pix[p]];
        int w = v + d - Q.k;
        w = w < 0 ? 0 : (w > 255 ? 255 : w);
        Q.dv[e] = w - v;
        if (Q.fold) Q.fxs[e] = __fdiv_rn((float)(w - v), 255.f);
    }
    if (Q.fold && threadIdx.x < Q.s) {  // the largest change of each pixel (steps -k and k, clipped)
        const int v = Q.image[Q.pix[threadIdx.x]];
        Q.fx[threadIdx.x] = __fdiv_ru((float)max(min(Q.k, 255 - v), min(Q.k, v)), 255.f);
    }
}

__device__ __forceinline__ double act64(int act, double u) {
    if (act == ACT_SIGMOID) return 1.0 / (1.0 + exp(-u));  // Eq. 2
    if (act == ACT_RELU) return u > 0.0 ? u : 0.0;
    return u;
}

// v / 255 of every grey level, FP64.
struct Grey {
    double v[256];
    constexpr Grey() : v() {
        for (int i = 0; i < 256; ++i) v[i] = (double)i / 255.0;
    }
};
__device__ constexpr Grey kGrey;

// Neuron i of layer l, WPN warps each; their lanes stride over the inputs. Also
// bounds the FP64 error of the result, in FP32 rounded up: a term passes at most
// c = K / lanes + 16 roundings (its lane's chain, the sums over lanes and warps, the
// bias; x / 255 on layer 1), so c 2^-53 (sum_j |w_j h_j| + |b|), plus the input errors
// propagated, sum_j |w_j| e_j (the activations are 1-Lipschitz).
//
// With Q.fold the warps also write their neuron's row of the folded net (fold.cu):
// du_i as a linear form in the s pixel changes and the sources of the nodes of
// earlier layers, the row of W_l times the rows of the layer below ("pos" inputs and
// nodes with ub >= 0, whose linear part is carried too), W_l itself in the columns of
// that layer's nodes; the bound B_i on |du_i| over the box; and the class that
// follows from it. Each block
// lists the layer below's "pos" neurons and nodes once, in order. A row's
// columns lie across a warp's lanes; fewer than 32 of them split the inputs too.
//
// Bound by load latency at the start, by FP64 after it: that pipe takes 16 cycles a
// warp instruction, so only the base product runs on it (2 instructions a term); rows
// are FP32 pairs (dfloat.cuh: 10 FP32 instructions against 32 cycles), bounds FP32.
// Few queries leave most of the chip idle with one warp per neuron (an output layer
// of 10 is 10 warps, each walking 512 inputs one load latency after the other), so
// wide layers take eight and an output layer 32; with many queries the warps come from
// them. One warp adds up its neuron's partial sums, the others go on to the columns
// (every warp adding them up kept the FP64 pipe busy for 3 to 4 us of each layer).
// The set-up of one query (init, layers, pack), at first (a warp per neuron, FP64
// throughout), with eight warps, and now: 784-512-512-10 142 -> 73 -> 60 us,
// 784-1024x3-10 310 -> 154 -> 106 us, 784-300-100-10 (80 ->) 51 us.
template <int WPN>
__global__ void __launch_bounds__(32 * (WPN > 8 ? WPN : 8)) k_pro_layer(NetView net, QueryView* qs, int nq, int l) {
    constexpr int NW = WPN > 8 ? WPN : 8;  // warps of a block
    constexpr int NPB = NW / WPN;          // neurons per block
    constexpr int LR = kMaxWidth / (32 * NW);  // rounds of the block's lanes over the widest layer
    constexpr int PS = WPN > 1 ? WPN : 1;
    __shared__ short plist[kMaxWidth], clist[kFoldMax];
    __shared__ int wpos[NW], wnode[NW];
    __shared__ float2 part[PS][32];
    __shared__ double pdot[PS][32];
    __shared__ float psum[4][PS][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wn = warp % WPN;  // warp of its neuron
    const int i = blockIdx.x * NPB + warp / WPN;
    const int tn = 32 * wn + lane, step = 32 * WPN;
    const int K = net.dims[l - 1], N = net.dims[l];
    if (blockIdx.y == 0 && i < N)  // the row of W_l comes in while the layer below is at work
        for (int j = 32 * tn; j < K; j += 32 * step)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(net.W[l] + (size_t)i * K + j));
    chain_wait();
    chain_next();
    const QueryView& Q = qs[blockIdx.y];
    const int offp = l >= 2 ? net.noff[l - 1] : 0;
    const bool fold = Q.fold != 0;
    int npos = 0, nnode = 0, nb = 0;  // the layer below: "pos" neurons, nodes; nodes of the layers below it
    bool rows = fold;                 // false: more nodes than a folded net holds
    if (fold && l >= 2) {
        const unsigned char* cls = Q.fcls + offp;
        unsigned mp[LR], mn[LR];
        int cp = 0, cn = 0;
#pragma unroll
        for (int e = 0; e < LR; ++e) {
            const int j = 32 * (warp * LR + e) + lane;
            const int c = j < K ? cls[j] : 1;
            mp[e] = __ballot_sync(0xffffffffu, c == 0 || c == 3);
            mn[e] = __ballot_sync(0xffffffffu, c >= 2);
            cp += __popc(mp[e]);
            cn += __popc(mn[e]);
        }
        if (lane == 0) {
            wpos[warp] = cp;
            wnode[warp] = cn;
        }
        for (int m = 1; m < l - 1; ++m) nb += Q.fst[2 + m];
        __syncthreads();
        int bp = 0, bn = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            if (w < warp) {
                bp += wpos[w];
                bn += wnode[w];
            }
            npos += wpos[w];
            nnode += wnode[w];
        }
        rows = nb + nnode <= kFoldMax;  // the same for every block (and for the layers above)
        if (rows) {
#pragma unroll
            for (int e = 0; e < LR; ++e) {
                const int j = 32 * (warp * LR + e) + lane;
                const unsigned below = (1u << lane) - 1u;
                if ((mp[e] >> lane) & 1u) plist[bp + __popc(mp[e] & below)] = (short)j;
                if ((mn[e] >> lane) & 1u) {
                    const int c = bn + __popc(mn[e] & below);
                    clist[c] = (short)j;
                    if (blockIdx.x == 0) Q.fnode[nb + c] = offp + j;
                }
                bp += __popc(mp[e]);
                bn += __popc(mn[e]);
            }
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            Q.fst[2 + l - 1] = nnode;
            if (!rows) Q.fst[1] = 1;
        }
        __syncthreads();
    }
    if (WPN == 1 && i >= N) return;  // (else one neuron per block, the grid has N)
    const float* Wr = net.W[l] + (size_t)i * K;
    double dot = 0.0;
    float b[4] = {0.f, 0.f, 0.f, 0.f};  // sum |w h|, sum |w| e; of the carried rows: sum |w| fer, sum |w| B
    if (l == 1) {
#pragma unroll 4
        for (int j = tn; j < K; j += step) {
            const float w = Wr[j];
            const int v = Q.image[j];
            dot = fma((double)w, kGrey.v[v], dot);
            b[0] = __fmaf_ru(fabsf(w), (float)v, b[0]);
        }
        b[0] = __fdiv_ru(b[0], 255.f);
    } else {
        const double* h = Q.hb + offp;
        const double* eh = Q.eub + offp;
        if (fold) {
            const float2* he = Q.fhe + offp;
#pragma unroll 4
            for (int j = tn; j < K; j += step) {
                const float w = Wr[j];
                const float2 m = he[j];
                dot = fma((double)w, h[j], dot);
                b[0] = __fmaf_ru(fabsf(w), m.x, b[0]);
                b[1] = __fmaf_ru(fabsf(w), m.y, b[1]);
            }
            if (rows) {
#pragma unroll 2
                for (int jj = tn; jj < npos; jj += step) {
                    const int j = plist[jj];
                    const float w = fabsf(Wr[j]);
                    b[2] = __fmaf_ru(w, Q.fer[offp + j], b[2]);
                    b[3] = __fmaf_ru(w, Q.fbd[offp + j], b[3]);
                }
            }
        } else {
#pragma unroll 4
            for (int j = tn; j < K; j += step) {
                const float w = Wr[j];
                dot = fma((double)w, h[j], dot);
                b[0] = __fmaf_ru(fabsf(w), __double2float_ru(fabs(h[j])), b[0]);
                b[1] = __fmaf_ru(fabsf(w), __double2float_ru(eh[j]), b[1]);
            }
        }
    }
    const int n = net.noff[l] + i;
    double u = 0.0;
    float eu = 0.f;
    if (WPN > 1) {  // the neuron's first warp adds up, in 4 chains
        pdot[wn][lane] = dot;
#pragma unroll
        for (int m = 0; m < 4; ++m) psum[m][wn][lane] = b[m];
        __syncthreads();
        if (wn == 0) {
            double d4[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) d4[c] = pdot[c % PS][lane];
#pragma unroll
            for (int w = 4; w < WPN; ++w) d4[w & 3] += pdot[w % PS][lane];
            dot = (d4[0] + d4[1]) + (d4[2] + d4[3]);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                b[m] = psum[m][0][lane];
#pragma unroll
                for (int w = 1; w < WPN; ++w) b[m] = __fadd_ru(b[m], psum[m][w][lane]);
            }
        }
    }
    if (wn == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            dot += __shfl_xor_sync(0xffffffffu, dot, o);
#pragma unroll
            for (int m = 0; m < 4; ++m) b[m] = __fadd_ru(b[m], __shfl_xor_sync(0xffffffffu, b[m], o));
        }
        const float bias = net.b[l][i];
        u = dot + (double)bias;
        // (activations add 2^-50 |u|)
        eu = __fmul_ru((float)((K + step - 1) / step + 17) * 0x1p-53f, __fadd_ru(b[0], fabsf(bias)));
        eu = __fmaf_ru(0x1p-50f, __double2float_ru(fabs(u)), __fadd_ru(eu, b[1]));
        eu = __fmul_ru(eu, 1.f + 0x1p-20f);
    }
    if (tn == 0) {
        const double h = (l < net.L) ? act64(net.act, u) : u;
        Q.ub[n] = u;
        Q.hb[n] = h;
        Q.eub[n] = (double)eu;
        if (fold) Q.fhe[n] = make_float2(__double2float_ru(fabs(h)), eu);
    }
    if (!rows) return;
    const int s = Q.s;
    float2* row = Q.fco + (size_t)n * Q.fstride;
    float B = 0.f;  // sum of |coefficient| x bound of its source (over lanes of the first warp)
    // the rows of the layer below carry errors fer; a pair sum over npos inputs adds at
    // most (6.5 npos + 20) 2^-48 sum_j |w_j| B_j (PairSum), and joining its parts over
    // lanes and warps, in at most 14 steps, 42 2^-48 of it: below (npos + 32) 2^-45
    const float er = l == 1 ? 0.f : __fmaf_ru((float)(npos + 32) * 0x1p-45f, b[3], b[2]);
    if (l == 1) {
        if (wn == 0 && lane < s) {
            const float w = Wr[Q.pix[lane]];
            row[lane] = make_float2(w, 0.f);
            B = __fmul_ru(fabsf(w), Q.fx[lane]);
        }
    } else {
        const int S = s + nb;
        const float2* prev = Q.fco + (size_t)offp * Q.fstride;
        for (int k0 = 0; k0 < S; k0 += 32) {
            int sp = 1;  // lanes per input: a power of two that holds the columns left
            while (sp < 32 && sp < S - k0) sp <<= 1;
            const int per = 32 / sp;
            const int k = k0 + (lane & (sp - 1)), g = wn * per + lane / sp, G = WPN * per;
            PairSum sum;
            if (k < S) {
                for (int jj = g; jj < npos; jj += kSettle * G) {
                    float w[kSettle];
                    float2 h[kSettle];
#pragma unroll
                    for (int e = 0; e < kSettle; ++e) {  // in flight together, also the last few
                        const bool in = jj + e * G < npos;
                        const int j = plist[in ? jj + e * G : jj];
                        w[e] = in ? Wr[j] : 0.f;
                        h[e] = prev[(size_t)j * Q.fstride + k];
                    }
#pragma unroll
                    for (int e = 0; e < kSettle; ++e) sum.add(w[e], h[e]);
                    sum.settle();
                }
            }
            float2 a = sum.a;
            for (int o = sp; o < 32; o <<= 1)
                a = df_add(a, make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o)));
            if (WPN > 1) {
                __syncthreads();
                part[wn][lane] = a;
                __syncthreads();
                if (wn == 0) {
                    float2 a4[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) a4[c] = part[c % PS][lane];
#pragma unroll
                    for (int w = 4; w < WPN; ++w) a4[w & 3] = df_add(a4[w & 3], part[w % PS][lane]);
                    a = df_add(df_add(a4[0], a4[1]), df_add(a4[2], a4[3]));
                }
            }
            if (wn == 0 && lane < sp && k < S) {
                row[k] = a;
                B = __fmaf_ru(abs_up(a), k < s ? Q.fx[k] : Q.fsb[Q.fnode[k - s]], B);
            }
        }
        if (wn == 0)
            for (int c = lane; c < nnode; c += 32) {
                const float w = Wr[clist[c]];
                row[S + c] = make_float2(w, 0.f);
                B = __fmaf_ru(fabsf(w), Q.fsb[offp + clist[c]], B);
            }
    }
    if (wn != 0) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) B = __fadd_ru(B, __shfl_xor_sync(0xffffffffu, B, o));
    if (lane == 0) {
        B = __fadd_ru(B, er);
        Q.fbd[n] = B;
        Q.fer[n] = er;
        // products of weights may pass FP32's range: an infinity or NaN in a row (or er) is
        // one in B too, times whatever its source's bound is, and the query does not fold
        if (!(B < kFoldBig) || !(eu < kFoldBig)) Q.fst[1] = 1;
        // a neuron keeps its sign, clear of the tie band, over the whole box
        if (l < net.L) {
            const bool keeps = fabs(u) > ((double)B + (double)eu) * (1.0 + 1e-6) + 4.0 * kTau;
            Q.fcls[n] = keeps ? (u >= 0.0 ? 0 : 1) : (u >= 0.0 ? 3 : 2);
            // a node's source is at most as far as its potential can cross 0
            Q.fsb[n] = fmaxf(0.f, __fadd_ru(__fsub_ru(B, __double2float_rd(fabs(u))), eu));
        }
    }
}

__global__ void k_pro_tables(NetView net, QueryView* qs, int nq) {
    const QueryView& Q = qs[blockIdx.y];
    const int e = blockIdx.x;  // e = p * R + d
    if (e >= Q.s * Q.R || folded(Q)) return;
    const int p = e / Q.R;
    const int H0 = net.dims[0], H1 = net.dims[1];
    const double step = (double)Q.dv[e] / 255.0;
    const float* W1 = net.W[1];
    const int col = Q.pix[p];
    for (int j = threadIdx.x; j < H1; j += blockDim.x)
        Q.tab[(size_t)e * H1 + j] = (float)((double)W1[(size_t)j * H0 + col] * step);
}

// Rounded-up float of a non-negative double.
__device__ __forceinline__ float up(double x) { return __double2float_ru(x); }

__device__ __forceinline__ double block_sum(double v, double* red) {
    // blockDim.x is a multiple of 32 and at most 1024
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) {
        t = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) red[32] = t;
    }
    __syncthreads();
    return red[32];
}

// Screen constants. With fl() the fp32 rounding and u = 2^-24:
//  dub_n   = |fl(ub_n) - ub_n| + eub_n   (+ e1_j on layer 1); eub bounds the FP64
//            error of ub itself, so every screen decision holds in exact arithmetic
//  thr_n   = dub_n + 2 tau, infinite when |ub_n| < tau (every evaluation of n is
//            a sign tie)
//  e1_j    = (gamma_{s+2} + 2u) * sum_p max_d |tab[p][d][j]|, the layer-1 table-sum error
//  ReLU:     c1 = 0, c2 = -fl(ub) when ub >= 0; c1 = fl(ub), c2 = 0 otherwise, so the
//            output change is max(du + c1, c2)
//  sigmoid / identity: c1 = fl(ub), c2 = fl(hb)
//  kvec[l] = norm of the point-independent part of the layer-l output error
__global__ void k_pro_finish(NetView net, QueryView* qs, int nq) {
    __shared__ double red[33];
    QueryView& Q = qs[blockIdx.x];
    if (folded(Q)) return;
    const int L = net.L, HL = net.dims[L];
    const double* y = Q.ub + net.noff[L];
    if (threadIdx.x == 0) {
        int D = 0;
        for (int i = 1; i < HL; ++i)
            if (y[i] > y[D]) D = i;
        double mx = -DBL_MAX;
        for (int i = 0; i < HL; ++i)
            if (i != D && y[i] > mx) mx = y[i];
        Q.cnt->D = D;
        // Eq. 10 margin, or max(y_D - V, V - max_{i!=D} y_i) for Eq. 11
        Q.cnt->base_margin = Q.prop == PROP_THRESHOLD ? fmax(y[D] - Q.V, Q.V - mx) : y[D] - mx;
    }
    const double u24 = 0x1p-24;
    const int s = Q.s;
    const double gam = (s + 2) * u24 / (1.0 - (s + 2) * u24) + 2.0 * u24;
    for (int l = 1; l <= L; ++l) {
        const int H = net.dims[l];
        double ss_a = 0.0, ss_b = 0.0;  // squared norms of per-neuron constant errors
        for (int i = threadIdx.x; i < H; i += blockDim.x) {
            const int n = net.noff[l] + i;
            const double ub = Q.ub[n], hb = Q.hb[n];
            const float ub32 = __double2float_rn(ub);
            const double dub = fabs((double)ub32 - ub) + Q.eub[n];
            double e1 = 0.0;
            if (l == 1) {
                double b1 = 0.0;
                // dv_p grows with the digit, so |tab| is largest at one of the ends
                for (int p = 0; p < s; ++p)
                    b1 += fmax(fabs((double)Q.tab[(size_t)p * Q.R * H + i]),
                               fabs((double)Q.tab[((size_t)p * Q.R + Q.R - 1) * H + i]));
                e1 = gam * b1 * (1.0 + 1e-12);
            }
            const bool base_tie = fabs(ub) < kTau;
            Q.ub32[n] = ub32;
            Q.dub[n] = up(dub + e1);
            Q.thr[n] = base_tie ? INFINITY : up(dub + e1 + 2.0 * kTau);
            if (net.act == ACT_RELU) {
                Q.c1[n] = ub >= 0.0 ? 0.0f : ub32;
                Q.c2[n] = ub >= 0.0 ? -ub32 : 0.0f;
            } else {
                Q.c1[n] = ub32;
                Q.c2[n] = __double2float_rn(hb);
            }
            const double dhb = fabs((double)__double2float_rn(hb) - hb) + Q.eub[n];
            if (l < L) {
                if (net.act == ACT_RELU) {
                    ss_a += (e1 + dub) * (e1 + dub);
                } else if (net.act == ACT_SIGMOID) {
                    ss_a += (e1 + dub) * (e1 + dub);
                    ss_b += dhb * dhb;
                } else {
                    ss_a += e1 * e1;
                }
            }
        }
        double na = sqrt(block_sum(ss_a, red));
        double nb = sqrt(block_sum(ss_b, red));
        if (threadIdx.x == 0) {
            double kv = 0.0;
            if (l < L) {
                if (net.act == ACT_RELU) kv = na;
                else if (net.act == ACT_SIGMOID) kv = 0.25 * na + nb + sqrt((double)H) * 8.0 * u24;
                else kv = na;
            }
            Q.kvec[l] = up(kv * (1.0 + 1e-9));
        }
        __syncthreads();
    }
}

// Time to verdict of queries whose work count never reached zero inside a pass
// (no screen tiles: empty ranges and the FP64-only path): the end of the last pass.
__global__ void k_stamp_final(QueryView* qs, int nq) {
    chain_wait();
    chain_next();
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nq) return;
    Counters* c = qs[q].cnt;
    if (c->t_final == 0) c->t_final = globaltimer_ns();
}

void launch_stamp_final(QueryView* d_qs, int nq, cudaStream_t st) {
    launch_chained(k_stamp_final, (nq + 127) / 128, 128, 0, st, d_qs, nq);
}

// Blocks per query that clear the result buffers: one for the small masks, more
// where a verdict bitmap makes them large (a single block of 256 threads clears
// 1.4 MB in about 40 us), fewer when many queries fill the chip by themselves.
static unsigned clear_blocks(int nq, unsigned long long max_hi) {
    const unsigned long long b = 1 + max_hi / (32ull * 4 * 256 * 4);
    const unsigned long long most = nq >= 64 ? 4 : 256 / (unsigned)nq;
    return (unsigned)(b < most ? b : most);
}

void launch_pro_init(const NetView& net, QueryView* d_qs, int nq, cudaStream_t st, unsigned long long max_hi) {
    launch_chained(k_pro_init, dim3((unsigned)nq, clear_blocks(nq, max_hi)), 256, 0, st, net, d_qs, nq);
}

void launch_pro_layer(const NetView& net, QueryView* d_qs, int nq, int l, cudaStream_t st) {
    // eight warps per neuron for at least 256 inputs (one round of their lanes), until
    // the queries alone put about 16 warps on every SM; where the neurons alone leave
    // most SMs empty (output layers of few queries) 32 of them, eight for few inputs
    constexpr long long kSms = 152;
    const long long neurons = (long long)nq * net.dims[l];
    if (net.dims[l - 1] >= 256 && neurons <= kSms)
        launch_chained(k_pro_layer<32>, dim3(net.dims[l], nq), 1024, 0, st, net, d_qs, nq, l);
    else if (neurons <= (net.dims[l - 1] >= 256 ? 16 * kSms : kSms))
        launch_chained(k_pro_layer<8>, dim3(net.dims[l], nq), 256, 0, st, net, d_qs, nq, l);
    else
        launch_chained(k_pro_layer<1>, dim3((net.dims[l] + 7) / 8, nq), 256, 0, st, net, d_qs, nq, l);
}

void launch_prologue(const NetView& net, QueryView* d_qs, int nq, cudaStream_t st, unsigned long long max_hi,
                     bool fold, unsigned long long* d_unfolded) {
    launch_pro_init(net, d_qs, nq, st, max_hi);
    for (int l = 1; l <= net.L; ++l) launch_pro_layer(net, d_qs, nq, l, st);
    if (fold) launch_fold_pack(net, d_qs, nq, st, d_unfolded);
}

void launch_prologue_screens(const NetView& net, QueryView* d_qs, int nq, int max_sr, cudaStream_t st) {
    if (max_sr > 0) k_pro_tables<<<dim3(max_sr, nq), 256, 0, st>>>(net, d_qs, nq);
    k_pro_finish<<<nq, 256, 0, st>>>(net, d_qs, nq);
}

}  // namespace vbmc
