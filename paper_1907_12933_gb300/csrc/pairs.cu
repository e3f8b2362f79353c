// pairs.cu -- the covering methods of Sec. III-B over a set of input pairs
// (x1, x2) without enumeration: potentials of both inputs (Eq. 1, the hidden
// activation on layers 1..L-1; FP64 with a CTA per pair in k_pairs, FP32 pairs with
// FP64 for undecided pairs in k_pairs_df), then per pair
//   sc(n)   sign change (sign(u) = 1 iff u >= 0)
//   vc(n)   no sign change and max(|u1|, |u2|) >= g min(|u1|, |u2|)
//   dc(k)   no sign change in layer k and ||u_k(x1) - u_k(x2)||_2 >= d
//   SS (i, j): i the only sign change of layer k and sc(j)      (pair bits)
//   SV (i, j): i the only sign change of layer k and vc(j)      (pair bits)
//   DS (k, j): dc(k) and sc(j)   (bit of neuron j of layer k+1; covers (any i, j))
//   DV (k, j): dc(k) and vc(j)
// ORed over all pairs into the caller's masks. Ties: a potential with |u| <
// 1e-9 in either input, a ratio test |max - g min| <= 1e-9 or a distance test
// |dist - d| <= 1e-9 is undecided; a pair that holds only under some
// resolution of the undecided tests goes to the tie mask.
#include "../../include/vbmc.h"
#include "dev.cuh"
#include "dfloat.cuh"
#include "launch.h"

#include <algorithm>
#include <cmath>
#include <vector>

namespace vbmc {
const NetView* net_view(const vbmc_net* net);
vbmc_status set_error(vbmc_status st, const char* msg);
void ss_covered(const NetView& v, const uint32_t* ss, std::vector<char>& cov);
}  // namespace vbmc

using namespace vbmc;

namespace {

constexpr int TP = 256;

__device__ __forceinline__ double act64p(int act, double u) {
    if (act == ACT_SIGMOID) return 1.0 / (1.0 + exp(-u));
    if (act == ACT_RELU) return u > 0.0 ? u : 0.0;
    return u;
}

struct PairOut {
    uint32_t *flip, *flip_tie, *ss, *ss_tie, *sv, *sv_tie, *ds, *ds_tie, *dv, *dv_tie;
};

// Potentials of layers l0..L into u, layer l0-1 already in u (l0 >= 2) or the
// input x (grey levels / 255, l0 = 1).
__device__ void forward64_from(const NetView& net, int l0, const uint8_t* x, double* u, double* h) {
    const int H0 = net.dims[0];
    if (l0 == 1) {
        for (int j = threadIdx.x; j < H0; j += blockDim.x) h[j] = (double)x[j] / 255.0;
        __syncthreads();
    }
    for (int l = l0; l <= net.L; ++l) {
        const int K = net.dims[l - 1], N = net.dims[l];
        const float* WT = net.WT[l];
        const double* in = l == 1 ? h : u + net.noff[l - 1];
        for (int i = threadIdx.x; i < N; i += blockDim.x) {
            double acc = (double)net.b[l][i];
            for (int j = 0; j < K; ++j) {
                const double hj = l == 1 ? in[j] : act64p(net.act, in[j]);
                acc = fma((double)WT[(size_t)j * N + i], hj, acc);
            }
            u[net.noff[l] + i] = acc;
        }
        __syncthreads();
    }
}

// Potentials of every non-input neuron for input x (grey levels / 255) into u.
__device__ void forward64(const NetView& net, const uint8_t* x, double* u, double* h) {
    forward64_from(net, 1, x, u, h);
}

// Shared scratch of one CTA: the two inputs' potentials and per-neuron flags.
struct PairScratch {
    double *u1, *u2, *h;
    unsigned char *fl, *ti, *vc, *vt;  // certain sign change, sign tie, certain value change, undecided
};

__device__ PairScratch pair_scratch(const NetView& net, double* sh) {
    const int total = net.total, H0 = net.dims[0];
    const int gw = H0 > net.hmax ? H0 : net.hmax;
    PairScratch P;
    P.u1 = sh;
    P.u2 = P.u1 + total;
    P.h = P.u2 + total;  // [gw]
    P.fl = reinterpret_cast<unsigned char*>(P.h + gw);
    P.ti = P.fl + total;
    P.vc = P.ti + total;
    P.vt = P.vc + total;
    return P;
}

// The covers of one pair from its potentials u1, u2 (all threads of the CTA).
__device__ void pair_covers(const NetView& net, const PairScratch& P, double g, double d, const PairOut& o) {
    __shared__ int nflip[kMaxL + 2], ntie[kMaxL + 2], only[kMaxL + 2];
    __shared__ double dist2[kMaxL + 2];
    const int total = net.total;
    const double tau = kTau;
    if (threadIdx.x <= kMaxL + 1) {
        nflip[threadIdx.x] = 0;
        ntie[threadIdx.x] = 0;
        only[threadIdx.x] = -1;
        dist2[threadIdx.x] = 0.0;
    }
    __syncthreads();
    for (int n = threadIdx.x; n < total; n += blockDim.x) {
        const double a1 = P.u1[n], a2 = P.u2[n];
        const bool t = fabs(a1) < tau || fabs(a2) < tau;
        const bool f = !t && ((a1 >= 0.0) != (a2 >= 0.0));
        const double a = fabs(a1), b = fabs(a2);
        const double test = fmax(a, b) - g * fmin(a, b);
        const bool v = !f && !t && test > tau;
        P.ti[n] = t;
        P.fl[n] = f;
        P.vc[n] = v;
        P.vt[n] = !f && !v && (t || fabs(test) <= tau);
        int l = 1;
        while (l < net.L && n >= net.noff[l + 1]) ++l;
        if (f) {
            atomicAdd(&nflip[l], 1);
            atomicMax(&only[l], n - net.noff[l]);
            if (o.flip) set_bit_once(o.flip, (unsigned long long)n);
        }
        if (t) {
            atomicAdd(&ntie[l], 1);
            if (o.flip_tie) set_bit_once(o.flip_tie, (unsigned long long)n);
        }
        const double e = a1 - a2;
        atomicAdd(&dist2[l], e * e);
    }
    __syncthreads();
    for (int l = 1; l < net.L; ++l) {
        const int Hl = net.dims[l], Hn = net.dims[l + 1], off = net.noff[l], on = net.noff[l + 1];
        const double dist = sqrt(dist2[l]);
        const bool dc_cert = nflip[l] == 0 && ntie[l] == 0 && dist - d > tau;
        const bool dc_poss = nflip[l] == 0 && dist - d >= -tau;
        for (int i = threadIdx.x; i < Hn; i += blockDim.x) {
            const int ni = on + i;
            const unsigned long long bit = (unsigned long long)ni;
            if (dc_cert && P.fl[ni]) { if (o.ds) set_bit_once(o.ds, bit); }
            else if (dc_poss && (P.fl[ni] || P.ti[ni])) { if (o.ds_tie) set_bit_once(o.ds_tie, bit); }
            if (dc_cert && P.vc[ni]) { if (o.dv) set_bit_once(o.dv, bit); }
            else if (dc_poss && (P.vc[ni] || P.vt[ni])) { if (o.dv_tie) set_bit_once(o.dv_tie, bit); }
        }
        // SS and SV: j the only changed neuron of layer l (for certain, or under ties)
        const int nf = nflip[l], nt = ntie[l], oj = only[l];
        for (int e = threadIdx.x; e < Hl * Hn; e += blockDim.x) {
            const int j = e / Hn, i = e % Hn;
            const bool certain = nt == 0 && nf == 1 && j == oj;
            const bool possible = certain || (nt > 0 && ((nf == 1 && j == oj) || (nf == 0 && P.ti[off + j])));
            if (!possible) continue;
            const int ni = on + i;
            const unsigned long long bit = (unsigned long long)net.ssoff[l] + (unsigned long long)j * Hn + i;
            if (certain && P.fl[ni]) { if (o.ss) set_bit_once(o.ss, bit); }
            else if (P.fl[ni] || P.ti[ni]) { if (o.ss_tie) set_bit_once(o.ss_tie, bit); }
            if (certain && P.vc[ni]) { if (o.sv) set_bit_once(o.sv, bit); }
            else if (P.vc[ni] || P.vt[ni]) { if (o.sv_tie) set_bit_once(o.sv_tie, bit); }
        }
    }
    __syncthreads();
}

__global__ void __launch_bounds__(TP) k_pairs(NetView net, const uint8_t* x1s, const uint8_t* x2s, int n_pairs,
                                               double g, double d, PairOut o) {
    extern __shared__ __align__(16) double sh[];
    const PairScratch P = pair_scratch(net, sh);
    const int H0 = net.dims[0];
    for (int p = blockIdx.x; p < n_pairs; p += gridDim.x) {
        forward64(net, x1s + (size_t)p * H0, P.u1, P.h);
        forward64(net, x2s + (size_t)p * H0, P.u2, P.h);
        pair_covers(net, P, g, d, o);
    }
}

// The same covers with the potentials as FP32 pairs (ReLU and identity nets). FP64
// runs at a sixty-fourth of the FP32 rate on this part and bound k_pairs; here a
// multiply-add costs five or six FP32 instructions. Every test a bit rests on (sign,
// value ratio, distance) has to clear its threshold by the potentials' error bound,
// else the CTA evaluates that pair in FP64 (k_pairs's own steps).
//
// A dot product against an anchor: a starts at sigma = 1.5 2^M, 2^(M-1) >= (1 + K 2^-22)
// ||W_i|| ||h||, so that no partial sum, the roundings included, leaves the binade
// [2^M, 2^(M+1)]; a' = fma(w, h, a) then rounds to the grid 2^(M-23), a - a' is exact, and
// r = fma(w, h, a - a') is what that step lost, summed plainly over 16 terms and then by
// two_sum. Per 16 terms the rests lose at most 136 2^(M-48), each rest 2^(M-48); with
// 2^M < 4 (1 + K 2^-22) ||W_i|| ||h||: |error| <= 5 (K + 16) 2^-45 ||W_i|| ||h||.
// Layer 1 runs on the grey levels (exact in FP32) and divides by 255 as a pair.
//
// CTA = IB images (IB / 2 pairs), a thread per neuron: one weight load serves IB
// images, whose activations are shared-memory broadcasts, high parts and low parts of
// an input side by side so that two images make one f32x2 operand: 4 (layer 1) or 5
// instructions for two multiply-adds. Layers stop where every pair is undecided. Bound by FP32 issue. 8,192 pairs on
// 784-512-512-10: FP64 55.5 ms, one image an instruction and a sum of its own 3.95 ms,
// now 3.45 ms (the kernel 2.87; its FMA pipe is 69 % busy, two cycles an f32x2).
constexpr int TPD = 256;

template <int IB>
struct PairDf {
    double dist2[IB / 2][kMaxL + 2];
    float E[IB], N[IB], X[IB];       // error norm and norm of a layer's input (layer 1: in grey levels);
    float M[IB];                     // 5 (K + 16) 2^-45 M + E with M the norm on the [0, 1] scale
    float sq[TPD / 32][IB / 2][4];   // per warp: ||h||^2 and ||u||^2 of a pair's two images
    double ds[TPD / 32][IB / 2];
    int nflip[IB / 2][kMaxL + 2], only[IB / 2][kMaxL + 2];
    int undec[IB / 2], differ[IB / 2];  // undecided; the two images differ
};

// K terms of neuron column w0 (stride N) against NP pairs of images, whose inputs start
// at in, row floats from one term to the next, the low parts lo floats behind the high ones.
template <int NP, bool L1>
__device__ __forceinline__ void anchored_dot(const float* __restrict__ w0, int N, int K, const float* in, int row,
                                             int lo, float sig, float2 (&u)[2 * NP]) {
    f32x2 A[NP], H[NP], Lo[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) {
        A[m] = pack2(sig, sig);
        H[m] = Lo[m] = 0ull;
    }
    f32x2 r[NP];
    auto term = [&](float w1, const float* h) {
        const f32x2 w = pack2(w1, w1);
        f32x2 hx[NP], hy[NP];
        if (NP % 2 == 0) {
#pragma unroll
            for (int m = 0; m < NP; m += 2) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(h + 2 * m);
                hx[m] = x.x;
                hx[(m + 1) % NP] = x.y;
                if (!L1) {
                    const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(h + lo + 2 * m);
                    hy[m] = y.x;
                    hy[(m + 1) % NP] = y.y;
                }
            }
        } else {
#pragma unroll
            for (int m = 0; m < NP; ++m) {
                hx[m] = *reinterpret_cast<const f32x2*>(h + 2 * m);
                if (!L1) hy[m] = *reinterpret_cast<const f32x2*>(h + lo + 2 * m);
            }
        }
#pragma unroll
        for (int m = 0; m < NP; ++m) {
            const f32x2 a = fma2(w, hx[m], A[m]);
            f32x2 e = fma2(w, hx[m], sub2(A[m], a));
            if (!L1) e = fma2(w, hy[m], e);
            r[m] = add2(r[m], e);
            A[m] = a;
        }
    };
    constexpr int KB = 16;
    float w[KB];  // a block's weights come in while the block before is at work
    const float* wp = w0;
    if (K >= KB) {
#pragma unroll
        for (int j = 0; j < KB; ++j) w[j] = __ldg(wp + (size_t)j * N);
    }
    for (int k0 = 0; k0 < K; k0 += KB) {
#pragma unroll
        for (int m = 0; m < NP; ++m) r[m] = 0ull;
        const float* h = in + (size_t)k0 * row;
        if (k0 + KB <= K) {
            float c[KB];
#pragma unroll
            for (int j = 0; j < KB; ++j) c[j] = w[j];
            wp += (size_t)KB * N;
            if (k0 + 2 * KB <= K) {
#pragma unroll
                for (int j = 0; j < KB; ++j) w[j] = __ldg(wp + (size_t)j * N);
            }
#pragma unroll
            for (int j = 0; j < KB; ++j) term(c[j], h + (size_t)j * row);
        } else {
#pragma unroll 1
            for (int j = 0; k0 + j < K; ++j) term(__ldg(w0 + (size_t)(k0 + j) * N), h + (size_t)j * row);
        }
#pragma unroll
        for (int m = 0; m < NP; ++m) {  // two_sum
            const f32x2 t = add2(H[m], r[m]), b = sub2(t, H[m]);
            Lo[m] = add2(Lo[m], add2(sub2(H[m], sub2(t, b)), sub2(r[m], b)));
            H[m] = t;
        }
    }
#pragma unroll
    for (int m = 0; m < NP; ++m) {
        const float2 a = unpack2(A[m]), h = unpack2(H[m]), l = unpack2(Lo[m]);
        u[2 * m] = df_add(make_float2(__fsub_rn(a.x, sig), 0.f), two_sum(h.x, l.x));
        u[2 * m + 1] = df_add(make_float2(__fsub_rn(a.y, sig), 0.f), two_sum(h.y, l.y));
    }
}

template <int IB>
__global__ void __launch_bounds__(TPD, 2) k_pairs_df(NetView net, const uint8_t* __restrict__ x1s,
                                                  const uint8_t* __restrict__ x2s, int n_pairs, double g, double d,
                                                  PairOut o, int bufw) {
    constexpr int PB = IB / 2;
    extern __shared__ __align__(16) double sh[];
    __shared__ PairDf<IB> T;
    // (16-byte reads in anchored_dot: rows of 2 IB floats, from a start that is aligned for them)
    float* const buf0 = reinterpret_cast<float*>(sh);   // [bufw][2][IB]: high parts, low parts
    float* const buf1 = buf0 + (size_t)bufw * 2 * IB;   // the same; layer 1's grey levels first
    unsigned char* const fl = reinterpret_cast<unsigned char*>(buf1 + (size_t)bufw * 2 * IB);  // [total][PB]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int H0 = net.dims[0], L = net.L;
    const bool relu = net.act == ACT_RELU;
    const float tau = __double2float_ru(kTau), gf = __double2float_ru(g);
    const float inv_hi = 1.f / 255.f;
    const float2 inv = make_float2(inv_hi, (float)(1.0 / 255.0 - (double)inv_hi));
    for (int p0 = blockIdx.x * PB; p0 < n_pairs; p0 += gridDim.x * PB) {
        const int np = min(PB, n_pairs - p0);
        float* const in0 = buf1;  // [H0][IB]
        if (tid < PB) T.differ[tid] = 0;
        __syncthreads();
        for (int im = 0; im < IB; ++im) {
            const uint8_t* x = (im & 1 ? x2s : x1s) + (size_t)(p0 + (im >> 1)) * H0;
            for (int k = tid; k < H0; k += TPD) {
                const float v = (im >> 1) < np ? (float)x[k] : 0.f;
                in0[k * IB + im] = v;
                if ((im & 1) && v != in0[k * IB + im - 1]) T.differ[im >> 1] = 1;
            }
        }
        if (tid < PB) T.undec[tid] = 0;
        for (int e = tid; e < PB * (kMaxL + 2); e += TPD) {
            T.nflip[e / (kMaxL + 2)][e % (kMaxL + 2)] = 0;
            T.only[e / (kMaxL + 2)][e % (kMaxL + 2)] = -1;
            T.dist2[e / (kMaxL + 2)][e % (kMaxL + 2)] = 0.0;
        }
        if (tid < IB) {  // grey levels: at most 255 sqrt(H_0)
            T.N[tid] = __fmul_ru(255.f, __fsqrt_ru((float)H0));
            T.E[tid] = 0.f;
        }
        __syncthreads();
        for (int l = 1; l <= L; ++l) {
            const int K = net.dims[l - 1], N = net.dims[l], off = net.noff[l];
            const float* in = l & 1 ? buf1 : buf0;
            float* const outb = l & 1 ? buf0 : buf1;
            const float* __restrict__ WT = net.WT[l];
            const float cK = 5.f * (float)(K + 16) * 0x1p-45f;
            float Nm = 0.f;
            for (int m = 0; m < IB; ++m) Nm = fmaxf(Nm, T.N[m]);
            Nm = __fmul_ru(Nm, __fmaf_ru((float)K, 0x1p-22f, 1.f));
            // sigma of a neuron: 1.5 2^M with 2^(M-1) >= (1 + K 2^-22) ||W_i|| max ||h|| (and above 0)
            auto anchor = [&](int n) {
                const int ex = ilogbf(fmaxf(__fmul_ru(net.rownorm[l][n], Nm), 1e-30f));
                return 1.5f * ldexpf(1.f, ex + 2);
            };
            // potentials: (sum) / 255 on layer 1, plus the bias
            auto finish = [&](float2 v, int n) {
                if (l == 1) {
                    const float p = __fmul_rn(v.x, inv.x);
                    float e = __fmaf_rn(v.x, inv.x, -p);
                    e = __fmaf_rn(v.x, inv.y, e);
                    e = __fmaf_rn(v.y, inv.x, e);
                    v = two_sum(p, e);
                }
                return df_add(v, make_float2(net.b[l][n], 0.f));
            };
            if (N * 4 >= TPD) {
                for (int n = tid; n < N; n += TPD) {
                    float2 u[IB];
                    if (l == 1) anchored_dot<PB, true>(WT + n, N, K, in, IB, 0, anchor(n), u);
                    else anchored_dot<PB, false>(WT + n, N, K, in, 2 * IB, IB, anchor(n), u);
#pragma unroll
                    for (int m = 0; m < IB; ++m) {
                        const float2 v = finish(u[m], n);
                        outb[(size_t)n * 2 * IB + m] = v.x;
                        outb[(size_t)n * 2 * IB + IB + m] = v.y;
                    }
                }
            } else {  // a narrow layer: a thread per neuron and pair
                for (int it = tid; it < N * PB; it += TPD) {
                    const int n = it / PB, pp = it % PB;
                    float2 u[2];
                    if (l == 1) anchored_dot<1, true>(WT + n, N, K, in + 2 * pp, IB, 0, anchor(n), u);
                    else anchored_dot<1, false>(WT + n, N, K, in + 2 * pp, 2 * IB, IB, anchor(n), u);
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        const float2 v = finish(u[m], n);
                        outb[(size_t)n * 2 * IB + 2 * pp + m] = v.x;
                        outb[(size_t)n * 2 * IB + IB + 2 * pp + m] = v.y;
                    }
                }
            }
            if (tid < IB) {  // layer 1: the input's norm and error on the [0, 1] scale
                const float nn = l == 1 ? __fmul_ru(T.N[tid], __fmul_ru(inv_hi, 1.f + 0x1p-22f)) : T.N[tid];
                T.M[tid] = nn;
                T.X[tid] = __fmaf_ru(cK, nn, T.E[tid]);
            }
            __syncthreads();
            // ---- the layer's tests, a thread per (neuron, pair); a thread keeps its pair
            const int pp = tid % PB;
            const float X1 = T.X[2 * pp], X2 = T.X[2 * pp + 1];
            const bool live = pp < np;
            // the value change counts where layer l - 1 has at most one sign change
            const bool ratio = l >= 2 && T.nflip[pp][l - 1] <= 1;
            float h1 = 0.f, h2 = 0.f, s1 = 0.f, s2 = 0.f;
            double dd = 0.0;
            for (int n = tid / PB; n < N; n += TPD / PB) {
                float2* const hi = reinterpret_cast<float2*>(outb + (size_t)n * 2 * IB + 2 * pp);
                float2* const lo = hi + IB / 2;
                const float2 uh = *hi, ul = *lo;
                const float2 a = make_float2(uh.x, ul.x), b = make_float2(uh.y, ul.y);
                if (live) {
                    const float rn = net.rownorm[l][n];
                    const float e1 = __fmaf_ru(rn, X1, __fmul_ru(0x1p-42f, fabsf(a.x)));
                    const float e2 = __fmaf_ru(rn, X2, __fmul_ru(0x1p-42f, fabsf(b.x)));
                    bool und = !(__fmul_rd(fabsf(a.x), 1.f - 0x1p-22f) > __fadd_ru(e1, tau)) ||
                               !(__fmul_rd(fabsf(b.x), 1.f - 0x1p-22f) > __fadd_ru(e2, tau));
                    const bool f = !und && ((a.x >= 0.f) != (b.x >= 0.f));
                    bool v = false;
                    if (ratio && !f && !und) {  // max - g min against tau
                        const float A = fabsf(a.x), B = fabsf(b.x), mx = fmaxf(A, B), mi = fminf(A, B);
                        const float t = fmaf(-(float)g, mi, mx);
                        const float et = __fadd_ru(__fmaf_ru(gf, fmaxf(e1, e2), fmaxf(e1, e2)), tau);
                        if (fabsf(t) > __fmaf_ru(0x1p-21f, __fmaf_ru(gf, mi, mx), et)) {
                            v = t > 0.f;
                        } else {  // near the threshold: the pairs' values in FP64
                            const double da = fabs((double)a.x + (double)a.y), db = fabs((double)b.x + (double)b.y);
                            const double td = fmax(da, db) - g * fmin(da, db);
                            if (fabs(td - kTau) <= (double)et || fabs(td + kTau) <= (double)et) und = true;
                            else v = td > kTau;
                        }
                    }
                    if (und) T.undec[pp] = 1;
                    if (f) {
                        atomicAdd(&T.nflip[pp][l], 1);
                        atomicMax(&T.only[pp][l], n);
                    }
                    fl[(size_t)(off + n) * PB + pp] = (unsigned char)((f ? 1 : 0) | (v ? 2 : 0));
                    const double df = ((double)a.x - (double)b.x) + ((double)a.y - (double)b.y);
                    dd += df * df;
                }
                s1 = __fmaf_ru(a.x, a.x, s1);
                s2 = __fmaf_ru(b.x, b.x, s2);
                if (l < L) {
                    if (relu) {
                        *hi = make_float2(fmaxf(a.x, 0.f), fmaxf(b.x, 0.f));
                        *lo = make_float2(a.x > 0.f ? a.y : 0.f, b.x > 0.f ? b.y : 0.f);
                    }
                    const float p = relu ? fmaxf(a.x, 0.f) : a.x, q = relu ? fmaxf(b.x, 0.f) : b.x;
                    h1 = __fmaf_ru(p, p, h1);
                    h2 = __fmaf_ru(q, q, h2);
                }
            }
#pragma unroll
            for (int x = PB; x < 32; x <<= 1) {
                h1 = __fadd_ru(h1, __shfl_xor_sync(0xffffffffu, h1, x));
                h2 = __fadd_ru(h2, __shfl_xor_sync(0xffffffffu, h2, x));
                s1 = __fadd_ru(s1, __shfl_xor_sync(0xffffffffu, s1, x));
                s2 = __fadd_ru(s2, __shfl_xor_sync(0xffffffffu, s2, x));
                dd += __shfl_xor_sync(0xffffffffu, dd, x);
            }
            if (lane < PB) {
                T.sq[warp][pp][0] = h1;
                T.sq[warp][pp][1] = h2;
                T.sq[warp][pp][2] = s1;
                T.sq[warp][pp][3] = s2;
                T.ds[warp][pp] = dd;
            }
            __syncthreads();
            if (tid < IB) {
                const int pq = tid >> 1, im = tid & 1;
                float hs = 0.f, us = 0.f;
                double ds = 0.0;
                for (int w = 0; w < TPD / 32; ++w) {
                    hs = __fadd_ru(hs, T.sq[w][pq][im]);
                    us = __fadd_ru(us, T.sq[w][pq][2 + im]);
                    ds += T.ds[w][pq];
                }
                // ||err(u_l)|| <= sigma_l E + 5 (K + 16) 2^-45 ||W_l||_F N + 2^-42 ||u||; the
                // activation is 1-Lipschitz (layer 1: its input carries no error)
                float En = __fmul_ru(__fmul_ru(cK, net.frob[l]), T.M[tid]);
                if (l > 1) En = __fmaf_ru(net.sig[l], T.E[tid], En);
                En = __fmul_ru(__fmaf_ru(0x1p-42f, __fsqrt_ru(us), En), 1.f + 0x1p-20f);
                const float other = __shfl_xor_sync((1u << IB) - 1u, En, 1);
                if (im == 0) {
                    T.dist2[pq][l] = ds;
                    // a layer without a sign change whose distance lies at an edge of the tie
                    // band around d: undecided (inside it the distance is a tie for certain; that
                    // of identical images is 0)
                    if (l < L && T.nflip[pq][l] == 0 && T.differ[pq]) {
                        const double dist = sqrt(ds), ed = (double)__fadd_ru(En, other) * 1.001 + 1e-12 * dist;
                        if (!(fabs(fabs(dist - d) - kTau) > ed)) T.undec[pq] = 1;
                    }
                }
                T.N[tid] = __fmul_ru(__fsqrt_ru(hs), 1.f + 0x1p-20f);
                T.E[tid] = En;
            }
            __syncthreads();
            bool left = false;  // a pair that is still decided
            for (int q = 0; q < np; ++q) left = left || !T.undec[q];
            if (!left) break;
        }
        // ---- covers: no sign is a tie in a decided pair, only a distance may be one
        for (int n = tid; n < net.total; n += TPD) {
            bool any = false;
            for (int q = 0; q < np; ++q) any = any || (!T.undec[q] && (fl[(size_t)n * PB + q] & 1));
            if (any && o.flip) set_bit_once(o.flip, (unsigned long long)n);
        }
        for (int q = 0; q < np; ++q) {
            if (T.undec[q]) continue;
            for (int l = 1; l < L; ++l) {
                const int nf = T.nflip[q][l];
                if (nf > 1) continue;
                const double over = nf == 0 ? sqrt(T.dist2[q][l]) - d : 0.0;
                if (!(over >= -kTau)) continue;
                uint32_t* const ds = over > kTau ? o.ds : o.ds_tie;
                uint32_t* const dv = over > kTau ? o.dv : o.dv_tie;
                const int Hn = net.dims[l + 1], on = net.noff[l + 1];
                const unsigned long long r0 = (unsigned long long)net.ssoff[l] + (unsigned long long)max(T.only[q][l], 0) * Hn;
                for (int i = tid; i < Hn; i += TPD) {
                    const unsigned char x = fl[(size_t)(on + i) * PB + q];
                    if (nf == 1) {
                        if ((x & 1) && o.ss) set_bit_once(o.ss, r0 + i);
                        if ((x & 2) && o.sv) set_bit_once(o.sv, r0 + i);
                    } else {
                        if ((x & 1) && ds) set_bit_once(ds, (unsigned long long)(on + i));
                        if ((x & 2) && dv) set_bit_once(dv, (unsigned long long)(on + i));
                    }
                }
            }
        }
        __syncthreads();
        // ---- the pairs left, in FP64
        unsigned left = 0;
        for (int q = 0; q < np; ++q) left |= (unsigned)(T.undec[q] != 0) << q;
        const PairScratch S = pair_scratch(net, sh);
        while (left) {
            const int q = __ffs(left) - 1;
            left &= left - 1u;
            __syncthreads();
            forward64(net, x1s + (size_t)(p0 + q) * H0, S.u1, S.h);
            forward64(net, x2s + (size_t)(p0 + q) * H0, S.u2, S.h);
            pair_covers(net, S, g, d, o);
        }
        __syncthreads();
    }
}

// The covers over the enumeration: the pairs (x, x_t) of the unperturbed image
// and each point t of [lo, hi) that passes the query's filter. x's potentials
// once per CTA; x_t's layer 1 incrementally from them (its s changed pixels),
// layers 2..L in full.
__global__ void __launch_bounds__(TP) k_enum_pairs(NetView net, QueryView Q, double g, double d, PairOut o,
                                                    unsigned long long* n_points) {
    extern __shared__ __align__(16) double sh[];
    const PairScratch P = pair_scratch(net, sh);
    __shared__ int dv[kMaxS];
    __shared__ int pass;
    const int H1 = net.dims[1];
    forward64(net, Q.image, P.u1, P.h);
    unsigned long long mine = 0;
    for (unsigned long long t = Q.lo + blockIdx.x; t < Q.hi; t += gridDim.x) {
        if (threadIdx.x == 0) {
            int dg[kMaxS];
            decode_digits(t, Q.s, Q.R, dg);
            long long s2 = 0;
            bool shell = Q.k == 0;
            for (int p = 0; p < Q.s; ++p) {
                const int v0 = Q.image[Q.pix_in[p]];
                int v1 = v0 + dg[p] - Q.k;
                v1 = v1 < 0 ? 0 : (v1 > 255 ? 255 : v1);
                dv[p] = v1 - v0;
                s2 += (long long)dv[p] * dv[p];
                shell = shell || dg[p] == 0 || dg[p] == Q.R - 1;
            }
            // the query's filter (the Euclidean ball of Eq. 9 on the grid, a k-shell)
            pass = (!(Q.filter & FILTER_L2) || s2 <= Q.l2max) && (!(Q.filter & FILTER_SHELL) || shell);
        }
        __syncthreads();
        if (!pass) {
            __syncthreads();
            continue;
        }
        ++mine;
        for (int j = threadIdx.x; j < H1; j += blockDim.x) {
            double a = P.u1[j];
            for (int p = 0; p < Q.s; ++p)
                a = fma((double)net.WT[1][(size_t)Q.pix_in[p] * H1 + j], (double)dv[p] / 255.0, a);
            P.u2[j] = a;
        }
        __syncthreads();
        forward64_from(net, 2, nullptr, P.u2, P.h);
        pair_covers(net, P, g, d, o);
    }
    if (threadIdx.x == 0 && mine) atomicAdd(n_points, mine);
}

}  // namespace

namespace vbmc {

// Clears the caller's masks and checks the cover parameters and the kernels'
// shared-memory need; sets *smem.
vbmc_status pair_setup(const NetView& v, const vbmc_cover_params* params, const vbmc_pair_masks* out,
                       cudaStream_t st, size_t* smem) {
    if (!(params->g >= 1.0) || !(params->d >= 0.0)) return set_error(VBMC_ERR_ARG, "need g >= 1 and d >= 0");
    const size_t fw = (size_t)v.flip_words * 4, sw = (size_t)v.ss_words * 4;
    uint32_t* const fmasks[6] = {out->flip, out->flip_tie, out->ds, out->ds_tie, out->dv, out->dv_tie};
    uint32_t* const smasks[4] = {out->ss, out->ss_tie, out->sv, out->sv_tie};
    for (uint32_t* m : fmasks)
        if (m && cudaMemsetAsync(m, 0, fw, st) != cudaSuccess) return set_error(VBMC_ERR_CUDA, "memset");
    for (uint32_t* m : smasks)
        if (m && sw && cudaMemsetAsync(m, 0, sw, st) != cudaSuccess) return set_error(VBMC_ERR_CUDA, "memset");
    const int gw = v.dims[0] > v.hmax ? v.dims[0] : v.hmax;
    *smem = sizeof(double) * (2 * (size_t)v.total + gw) + 4 * (size_t)v.total;
    if (*smem > 200 * 1024) return set_error(VBMC_ERR_UNSUPPORTED, "net too large for the pair kernel");
    return VBMC_OK;
}

int pair_grid(unsigned long long units) {
    int n_sm = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const unsigned long long cap = (unsigned long long)n_sm * 4;
    return (int)(units < cap ? units : cap);
}

// The covers over the pairs (unperturbed image, point) of the view's range;
// adds the points that pass the filter to *d_npoints.
vbmc_status launch_enum_pairs(const NetView& v, const QueryView& q, const vbmc_cover_params* params,
                              const vbmc_pair_masks* out, unsigned long long* d_npoints, cudaStream_t st) {
    size_t smem = 0;
    vbmc_status s = pair_setup(v, params, out, st, &smem);
    if (s != VBMC_OK) return s;
    if (q.hi <= q.lo) return VBMC_OK;
    cudaFuncSetAttribute(k_enum_pairs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const PairOut o{out->flip, out->flip_tie, out->ss, out->ss_tie, out->sv, out->sv_tie,
                    out->ds, out->ds_tie, out->dv, out->dv_tie};
    k_enum_pairs<<<pair_grid(q.hi - q.lo), TP, smem, st>>>(v, q, params->g, params->d, o, d_npoints);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? VBMC_OK : set_error(VBMC_ERR_CUDA, cudaGetErrorString(e));
}

}  // namespace vbmc

extern "C" vbmc_status vbmc_pair_coverage(const vbmc_net* net, const uint8_t* d_images1, const uint8_t* d_images2,
                                          int32_t n_pairs, const vbmc_cover_params* params,
                                          const vbmc_pair_masks* out, void* stream) {
    if (!net || !params || !out || (n_pairs > 0 && (!d_images1 || !d_images2)))
        return set_error(VBMC_ERR_ARG, "null argument");
    if (n_pairs < 0) return set_error(VBMC_ERR_ARG, "n_pairs must be >= 0");
    const NetView& v = *net_view(net);
    cudaStream_t st = (cudaStream_t)stream;
    size_t smem = 0;
    vbmc_status s = pair_setup(v, params, out, st, &smem);
    if (s != VBMC_OK || n_pairs == 0) return s;
    const PairOut o{out->flip, out->flip_tie, out->ss, out->ss_tie, out->sv, out->sv_tie,
                    out->ds, out->ds_tie, out->dv, out->dv_tie};
    // FP32 pairs where the activation has a pair form, 8 images per CTA once that still
    // gives every SM a CTA, else 2 (more CTAs, shorter chains per CTA). A dead neuron is a
    // sign tie in every pair, so none would be decided: FP64 at once, a CTA per pair (700 pairs
    // on 784-512-512-10 5.2 ms, 8.5 by way of FP32 pairs, whose CTAs hold 4 pairs each; 8,192
    // on 25-10-5 0.23 and 0.45 ms)
    const int bufw = std::max(v.hmax, (v.dims[0] + 1) / 2);
    auto df_smem = [&](int ib) {
        const size_t need = 2 * sizeof(float2) * (size_t)bufw * ib + (size_t)v.total * (ib / 2);
        return std::max(need, smem);
    };
    int n_sm = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const int ib = n_pairs >= 4 * n_sm && df_smem(8) <= 200 * 1024 ? 8 : 2;
    if (v.act != ACT_SIGMOID && !v.dead && df_smem(ib) <= 200 * 1024) {
        const size_t sm = df_smem(ib);
        const unsigned long long groups = ((unsigned long long)n_pairs + ib / 2 - 1) / (ib / 2);
        const unsigned grid = (unsigned)std::min<unsigned long long>(groups, (unsigned long long)n_sm * 8);
        auto kern = ib == 8 ? k_pairs_df<8> : k_pairs_df<2>;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        kern<<<grid, TPD, sm, st>>>(v, d_images1, d_images2, n_pairs, params->g, params->d, o, bufw);
    } else {
        cudaFuncSetAttribute(k_pairs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_pairs<<<pair_grid((unsigned long long)n_pairs), TP, smem, st>>>(v, d_images1, d_images2, n_pairs, params->g,
                                                                        params->d, o);
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? VBMC_OK : set_error(VBMC_ERR_CUDA, cudaGetErrorString(e));
}

extern "C" vbmc_status vbmc_covered_fraction(const vbmc_net* net, int32_t layout, const uint32_t* mask,
                                             double* fraction) {
    if (!net || !mask || !fraction) return set_error(VBMC_ERR_ARG, "null argument");
    if (layout != VBMC_LAYOUT_PAIRS && layout != VBMC_LAYOUT_LAYER)
        return set_error(VBMC_ERR_ARG, "layout must be VBMC_LAYOUT_PAIRS or VBMC_LAYOUT_LAYER");
    const NetView& v = *net_view(net);
    std::vector<char> cov((size_t)v.total, 0);
    if (layout == VBMC_LAYOUT_PAIRS) {
        ss_covered(v, mask, cov);
    } else {
        auto bit = [&](unsigned long long b) { return (mask[b >> 5] >> (b & 31)) & 1u; };
        for (int l = 1; l < v.L; ++l) {
            const int Hl = v.dims[l], Hn = v.dims[l + 1], off = v.noff[l], on = v.noff[l + 1];
            bool any = false;  // a covered neuron of layer l + 1 covers all of layer l
            for (int i = 0; i < Hn; ++i)
                if (bit((unsigned long long)(on + i))) {
                    cov[on + i] = 1;
                    any = true;
                }
            for (int j = 0; any && j < Hl; ++j) cov[off + j] = 1;
        }
    }
    long c = 0;
    for (char x : cov) c += x;
    *fraction = v.total ? (double)c / (double)v.total : 0.0;
    return VBMC_OK;
}
