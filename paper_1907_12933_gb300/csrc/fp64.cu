// fp64.cu -- the final pass: points evaluated in FP64 on CUDA cores.
//
// One CTA per point. Layer 1 is incremental (ub_1 + sum_p W_1[:, p] dv_p / 255,
// Eq. 1), layers 2..L are full FP64 dot products over W_l^T (coalesced), the
// hidden outputs use sigmoid (Eq. 2) or ReLU. The point's results follow the
// definitions directly:
//   * margin m = y_D - max_{i != D} y_i; |m| < tau: tie (listed, not counted);
//     otherwise adversarial iff argmax(y) (lowest index) != D      (Eq. 10)
//   * sign(u) = [u >= 0]; neuron n is a sign tie at this point when |u_n| < tau
//     or |ub_n| < tau; a non-tie sign change sets its flip bit, a sign tie
//     sets its flip-tie bit                                         (Sec. III-B)
//   * SS-Cover of (j in layer l, i in layer l+1): certain when layer l has no
//     tie and exactly one change (j) and i changes without tie; pairs that
//     hold only under some resolution of the ties go to the SS-tie mask.
//
// A range has a CTA per point. Queued points are mostly few, and one CTA is bound by its SM's
// FP64 pipe (16 cycles a warp instruction: two layers of 1024 take 1.3 ms), so a cluster
// of CL CTAs shares a point: a layer's neurons are dealt to the cluster's warps, their
// outputs go to every CTA's shared memory, and the first CTA does the rest. A weight
// becomes FP64 by its bits, not on that pipe. The sums keep their order. One queued
// point of 784-1024x3-10: 1,375 -> 380 us, now bound by the chain of dependent FP64 sums
// (weights loaded a block ahead: 380 us too, and ranges of small nets 11.1 -> 16.6 ms).
// A queue that holds more points than the launch has clusters fills the chip with a CTA
// per point: a dead neuron or two equal outputs send every point here, and clusters then
// wait at their barriers more than they compute (whole calls, 4,913 such points on 25-10-5
// 1,700 us by clusters, 430 a CTA each; on 784-512-512-10, sigmoid, 19.2 and 8.2 ms; 289
// points on it 1,730 and 1,200 us).
#include "dev.cuh"
#include "launch.h"

#include <cfloat>

namespace vbmc {
namespace {

constexpr int T64 = 256;

__device__ __forceinline__ double act64(int act, double u) {
    if (act == ACT_SIGMOID) return 1.0 / (1.0 + exp(-u));
    if (act == ACT_RELU) return u > 0.0 ? u : 0.0;
    return u;
}

// (double)w of an FP32 number by its bits; zero, subnormal and non-finite ones by conversion.
__device__ __forceinline__ double widen(float w) {
    const unsigned b = __float_as_uint(w);
    if (((b >> 23) & 255u) - 1u >= 254u) return (double)w;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}

// *p of CTA rank's shared memory = v.
__device__ __forceinline__ void store_cluster(double* p, unsigned rank, double v) {
    unsigned a = (unsigned)__cvta_generic_to_shared(p), ra;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
}

template <int CL>
__global__ void __launch_bounds__(T64)
k_fp64(NetView net, const QueryView* __restrict__ qs, const QEntry* __restrict__ gather,
       const unsigned long long* __restrict__ gather_count, unsigned long long gather_cap,
       unsigned long long range_lo, unsigned long long range_hi) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int total = net.total, hmax = net.hmax;
    double* u = reinterpret_cast<double*>(smem_raw);       // [total]
    constexpr int HB = CL > 1 ? 2 : 1;
    double* h0 = u + total;                                  // [HB][hmax]: layer l's outputs in l % HB
    unsigned char* fl = reinterpret_cast<unsigned char*>(h0 + HB * hmax);  // [total]
    unsigned char* ti = fl + total;                                         // [total]
    __shared__ int nflip[kMaxL + 2], ntie[kMaxL + 2], only[kMaxL + 2];
    __shared__ double dstep[kMaxS];
    __shared__ int skip;

    unsigned long long n;
    if (gather) {
        n = *gather_count;
        if (n > gather_cap) n = gather_cap;
    } else {
        n = range_hi - range_lo;
    }
    const int L = net.L;
    // more points than clusters: a CTA per point after all (the same choice in every CTA)
    const bool solo = CL == 1 || n > gridDim.x / CL;
    const unsigned parts = solo ? 1u : CL, rank = solo ? 0u : cluster_rank();
    if (!solo && n > 0) cluster_barrier();  // every CTA of the cluster has started
    for (unsigned long long e = blockIdx.x / parts; e < n; e += gridDim.x / parts) {
        unsigned long long t;
        int qi;
        if (gather) {
            QEntry en = gather[e];
            t = en.t;
            qi = (int)en.q;
        } else {
            t = range_lo + e;
            qi = 0;
        }
        const QueryView& Q = qs[qi];
        if (threadIdx.x == 0) {
            int d[kMaxS];
            decode_digits(t, Q.s, Q.R, d);
            for (int p = 0; p < Q.s; ++p) dstep[p] = (double)Q.dv[p * Q.R + d[p]] / 255.0;
            skip = !gather && Q.filter && !in_filter(Q, d);  // outside the L2 ball / shell
            if (!gather && Q.filter && !skip) atomicAdd(&Q.cnt->n_points, 1ull);
        }
        __syncthreads();
        const bool out = skip;
        if (threadIdx.x <= kMaxL + 1) {
            nflip[threadIdx.x] = 0;
            ntie[threadIdx.x] = 0;
            only[threadIdx.x] = -1;
        }
        __syncthreads();
        if (out) continue;  // every thread has read skip before the next point's overwrites it
        // layer 1, incremental in FP64
        {
            const int H0 = net.dims[0], H1 = net.dims[1];
            const float* W1 = net.W[1];
            for (int j = threadIdx.x; j < H1; j += T64) {
                double a = Q.ub[j];
                for (int p = 0; p < Q.s; ++p) a += (double)W1[(size_t)j * H0 + Q.pix[p]] * dstep[p];
                u[j] = a;
                h0[(1 % HB) * hmax + j] = (L > 1) ? act64(net.act, a) : a;
            }
        }
        __syncthreads();
        for (int l = 2; l <= L; ++l) {
            const int K = net.dims[l - 1], N = net.dims[l];
            const float* __restrict__ WT = net.WT[l];
            const float* b = net.b[l];
            const int off = net.noff[l];
            const double* h = h0 + (size_t)((l - 1) % HB) * hmax;
            double* const hn = h0 + (size_t)(l % HB) * hmax;
            // 32 neurons a warp, the point's CTAs in turn
            for (int i = (int)((threadIdx.x >> 5) * parts + rank) * 32 + (int)(threadIdx.x & 31); i < N;
                 i += (int)(T64 * parts)) {
                double a = 0.0;
#pragma unroll 16
                for (int j = 0; j < K; ++j) a += widen(__ldg(WT + (size_t)j * N + i)) * h[j];
                const double v = a + (double)b[i];
                if (solo) {
                    u[off + i] = v;
                    if (HB > 1 && l < L) hn[i] = act64(net.act, v);
                } else {
                    store_cluster(u + off + i, 0u, v);
                    if (l < L) {
                        const double y = act64(net.act, v);
                        for (unsigned c = 0; c < CL; ++c) store_cluster(hn + i, c, y);
                    }
                }
            }
            if (!solo) {
                cluster_barrier();
            } else {
                __syncthreads();
                if (HB == 1) {  // layer l's outputs take the place of its inputs
                    if (l < L)
                        for (int i = threadIdx.x; i < N; i += T64) hn[i] = act64(net.act, u[off + i]);
                    __syncthreads();
                }
            }
        }
        if (rank == 0) {
            // signs, ties, changes
            for (int nn = threadIdx.x; nn < total; nn += T64) {
                const double ub = Q.ub[nn], ut = u[nn];
                const bool tie = fabs(ut) < kTau || fabs(ub) < kTau;
                const bool ch = ((ut >= 0.0) != (ub >= 0.0)) && !tie;
                fl[nn] = ch;
                ti[nn] = tie;
                int l = 1;
                while (l < L && nn >= net.noff[l + 1]) ++l;
                if (ch) {
                    atomicAdd(&nflip[l], 1);
                    atomicMax(&only[l], nn - net.noff[l]);
                    if (Q.flip) set_bit_once(Q.flip, nn);
                }
                if (tie) {
                    atomicAdd(&ntie[l], 1);
                    if (Q.flip_tie) set_bit_once(Q.flip_tie, nn);
                }
            }
            __syncthreads();
            // SS-Cover pairs (j in l, i in l+1)
            if (Q.ss) {
                for (int l = 1; l < L; ++l) {
                    const int Hl = net.dims[l], Hn = net.dims[l + 1];
                    const int ol = net.noff[l], on = net.noff[l + 1];
                    const bool certain = ntie[l] == 0 && nflip[l] == 1;
                    if (!certain && ntie[l] == 0) continue;  // no flip or >= 2 certain flips
                    if (!certain && nflip[l] >= 2) continue;
                    for (int j = 0; j < Hl; ++j) {
                        bool cand;
                        if (certain || nflip[l] == 1) cand = (j == only[l]);
                        else cand = ti[ol + j];  // no certain flip, some ties: each tie may be the one
                        if (!cand) continue;
                        for (int i = threadIdx.x; i < Hn; i += T64) {
                            const unsigned long long bit = (unsigned long long)net.ssoff[l] +
                                                           (unsigned long long)j * Hn + i;
                            if (certain && fl[on + i]) set_bit_once(Q.ss, bit);
                            else if (fl[on + i] || ti[on + i]) set_bit_once(Q.ss_tie, bit);
                        }
                    }
                }
            }
            // verdict
            if (threadIdx.x == 0) {
                const int HL = net.dims[L];
                const double* y = u + net.noff[L];
                const int D = Q.cnt->D;
                int am = 0;
                double mx = -DBL_MAX;
                for (int i = 0; i < HL; ++i) {
                    if (y[i] > y[am]) am = i;
                    if (i != D && y[i] > mx) mx = y[i];
                }
                // Eq. 10: m = y_D - max_{i!=D} y_i; Eq. 11: m = max(y_D - V, V - max_{i!=D} y_i),
                // negative iff y_D < V < some other output
                const bool thr = Q.prop == PROP_THRESHOLD;
                const double m = thr ? fmax(y[D] - Q.V, Q.V - mx) : y[D] - mx;
                if (thr) am = m < 0.0 ? -1 : D;
                if (fabs(m) < kTau) {
                    unsigned long long k = atomicAdd(&Q.cnt->n_ties, 1ull);
                    if (k < Q.ties_cap) Q.ties[k] = t;
                    else atomicOr(&Q.cnt->err, DERR_TIES);
                } else if (am != D) {
                    record_adversarial(Q, t);
                }
                if (gather) work_done(Q.cnt, 1);  // time to verdict: this queued point is resolved
            }
        }
        if (solo) __syncthreads();
        else cluster_barrier();  // the first CTA has read what the next point's layers write
    }
}

// Potential i of layer l at the point whose pixel changes are the lanes' x (lane p: pixel
// p's dv / 255), from layer l - 1's outputs h: a warp, its lanes over the inputs, so that a
// sum passes K / 32 + 6 roundings.
__device__ __forceinline__ double warp_potential(const NetView& net, const QueryView& Q, int l, int i, double x,
                                                 const double* h) {
    const int lane = threadIdx.x & 31, K = net.dims[l - 1];
    double a = 0.0;
    if (l == 1) {
        if (lane < Q.s) a = (double)net.W[1][(size_t)i * K + Q.pix[lane]] * x;
    } else {
        const float* w = net.W[l] + (size_t)i * K;
#pragma unroll 8
        for (int j = lane; j < K; j += 32) a = fma(widen(__ldg(w + j)), h[j], a);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a + (l == 1 ? Q.ub[i] : (double)net.b[l][i]);
}

// dv / 255 of pixel `lane` at point t.
__device__ __forceinline__ double lane_change(const QueryView& Q, unsigned long long t) {
    int d[kMaxS];
    decode_digits(t, Q.s, Q.R, d);
    double x = 0.0;
    for (int p = 0; p < Q.s; ++p)
        if ((int)(threadIdx.x & 31) == p) x = (double)Q.dv[p * Q.R + d[p]] / 255.0;
    return x;
}

// Outputs of hidden layer l at point t of query 0 into out, a warp per neuron.
__global__ void __launch_bounds__(T64) k_margin_layer(NetView net, const QueryView* qs, int l, unsigned long long t,
                                                      const double* h, double* out) {
    const int i = blockIdx.x * (T64 / 32) + (threadIdx.x >> 5);
    chain_wait();
    chain_next();
    if (i >= net.dims[l]) return;
    const QueryView& Q = qs[0];
    const double u = warp_potential(net, Q, l, i, l == 1 ? lane_change(Q, t) : 0.0, h);
    if ((threadIdx.x & 31) == 0) out[i] = act64(net.act, u);
}

// The output layer, and the FP64 margin: y_D - max_{i != D} y_i (Eq. 10), or Eq. 11's.
__global__ void __launch_bounds__(1024) k_margin_out(NetView net, const QueryView* qs, unsigned long long t,
                                                     const double* h, double* out) {
    __shared__ double y[kMaxWidth];
    chain_wait();
    const QueryView& Q = qs[0];
    const int L = net.L, HL = net.dims[L];
    const double x = L == 1 ? lane_change(Q, t) : 0.0;
    for (int i = threadIdx.x >> 5; i < HL; i += 32) {
        const double u = warp_potential(net, Q, L, i, x, h);
        if ((threadIdx.x & 31) == 0) y[i] = u;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int D = Q.cnt->D;
    double mx = -DBL_MAX;
    for (int i = threadIdx.x; i < HL; i += 32)
        if (i != D && y[i] > mx) mx = y[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (threadIdx.x == 0) *out = Q.prop == PROP_THRESHOLD ? fmax(y[D] - Q.V, Q.V - mx) : y[D] - mx;
}

}  // namespace

void launch_margin64(const NetView& net, const QueryView* d_qs, unsigned long long t, double* d_out,
                     cudaStream_t st) {
    // a launch per layer, its neurons over the chip. The getter's whole call: 784-512-512-10
    // 38 us, 784-1024x3-10 53 us (one CTA that walks the whole net, a thread per neuron: the
    // kernel alone 239, the call 1,286; the rows of a folded net, in FP32 pairs: 63)
    double* const h = d_out + 1;
    for (int l = 1; l < net.L; ++l)
        launch_chained(k_margin_layer, (net.dims[l] + T64 / 32 - 1) / (T64 / 32), T64, 0, st, net, d_qs, l, t,
                       h + (size_t)((l - 1) & 1) * net.hmax, h + (size_t)(l & 1) * net.hmax);
    launch_chained(k_margin_out, 1, 1024, 0, st, net, d_qs, t, h + (size_t)((net.L - 1) & 1) * net.hmax, d_out);
}

void launch_fp64(const NetView& net, const QueryView* d_qs, int nq, const QEntry* gather,
                 const unsigned long long* gather_count, unsigned long long gather_cap,
                 unsigned long long range_lo, unsigned long long range_hi, int n_sm,
                 cudaStream_t st) {
    // 8 CTAs per SM, most of them resident: with 6 or 4 the last points of a long queue leave
    // the chip idle (25-10-5, 83,521 points: 5.0 ms, 5.3 with 6; sigmoid 784-512-512-10,
    // 4,913 points: 8.2 ms, 9.0 with 4)
    constexpr int CL = 8, kGatherCtas = 8;
    auto smem = [&](int buffers) { return sizeof(double) * (net.total + buffers * (size_t)net.hmax) + 2 * (size_t)net.total; };
    if (gather && smem(2) <= 200 * 1024 && n_sm * kGatherCtas >= CL) {
        cudaFuncSetAttribute(k_fp64<CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem(2));
        cudaLaunchConfig_t c{};
        c.gridDim = (unsigned)(n_sm * kGatherCtas / CL * CL);
        c.blockDim = T64;
        c.dynamicSmemBytes = smem(2);
        c.stream = st;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = CL;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        c.attrs = &at;
        c.numAttrs = 1;
        cudaLaunchKernelEx(&c, k_fp64<CL>, net, d_qs, gather, gather_count, gather_cap, range_lo, range_hi);
        return;
    }
    cudaFuncSetAttribute(k_fp64<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem(1));
    unsigned grid = (unsigned)n_sm * 8;
    if (!gather) {
        const unsigned long long n = range_hi - range_lo;
        if (n < grid) grid = (unsigned)(n ? n : 1);
    }
    k_fp64<1><<<grid, T64, smem(1), st>>>(net, d_qs, gather, gather_count, gather_cap, range_lo, range_hi);
}

}  // namespace vbmc
