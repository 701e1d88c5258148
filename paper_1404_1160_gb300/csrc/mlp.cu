// mlp.cu -- the network of the learned stepper: a 5-64-64-2 GELU perceptron
// with bfloat16 weights and FP32 accumulation, its 64 x 64 products on the
// 5th-generation tensor cores (tcgen05.mma, bf16 x bf16 -> f32 in tensor
// memory) for inference, the learned step's correction and training.  The paper has no
// learned component; the network corrects one macro step of the improved ETD
// scheme (Algorithm ETDFSSModAlgo) and is defined, with its rounding points,
// as:
//
//   x = (r, v, sin(t/eps), cos(t/eps), dt)
//   z1 = W1 x + b1,   h1 = gelu(z1)                 (CUDA cores, FP32)
//   z2 = W2 bf16(h1) + b2,  h2 = gelu(z2)           (tensor cores)
//   out = W3 bf16(h2) + b3                          (CUDA cores, FP32)
//
// W1, W2, W3 are the bfloat16 roundings of FP32 master weights; gelu(u) =
// u erfc(-u / sqrt 2) / 2.  Training minimises sum((out - y)^2) / (2B) with
// Adam on the master weights.  Backward:
//   dout = (out - y) / B, dW3 = dout^T bf16(h2), db3 = sum dout,
//   dz2 = (dout W3) gelu'(z2), dW2 = bf16(dz2)^T bf16(h1), db2 = sum dz2,
//   dz1 = (bf16(dz2) W2) gelu'(z1), dW1 = dz1^T x, db1 = sum dz1.
// One kernel takes a tile of 128 samples through forward, backward and the
// tile's weight gradients (dW2 on the tensor cores, the samples as the
// reduction dimension) into per-block partials; a second one sums them in a
// fixed order, applies Adam and refreshes the rounded copies, so training is
// reproducible bit for bit.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "energy_check.cuh"
#include "gelu_fast.cuh"
#include "pic_internal.h"
#include "tc_desc.cuh"

namespace pic {

// flat parameter layout (FP32 masters)
constexpr int kMIn = 5, kMHid = 64, kMOut = 2;
constexpr int oW1 = 0, ob1 = oW1 + kMHid * kMIn, oW2 = ob1 + kMHid, ob2 = oW2 + kMHid * kMHid, oW3 = ob2 + kMHid,
              ob3 = oW3 + kMOut * kMHid, kMParams = ob3 + kMOut;
static_assert(kMParams == 4674, "parameter count");
// compact FP32 block used by the CUDA-core layers: bf16-rounded W1 and W3, biases
constexpr int sW1 = 0, sb1 = sW1 + kMHid * kMIn, sb2 = sb1 + kMHid, sW3 = sb2 + kMHid, sb3 = sW3 + kMOut * kMHid,
              kMSmall = sb3 + kMOut;

constexpr int kLossHist = 4096;   // batch losses kept on the device between copies to the host

struct MlpDev {
    float *master, *m, *v;
    __nv_bfloat16* W2b;   // [j][k]
    __nv_bfloat16* W2Tb;  // [k][j]
    float* small;         // kMSmall
    float* loss_part;     // per training block
    float* grad_part;     // [training blocks][kMParams]
    float* grad;          // [kMParams]
    float* loss;          // [kLossHist]
    int* err;             // set by a tensor-core wait that ran out of time (pinned host memory, mapped)
};

// ------------------------------------------------------------ device math

__device__ __forceinline__ float gelu_d(float u) {
    return 0.5f * erfcf(-u * 0.70710678118654752f) + u * 0.39894228040143268f * expf(-0.5f * u * u);
}
__device__ __forceinline__ unsigned int pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<unsigned int*>(&v);
}
__device__ __forceinline__ float round_bf16(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// Sample index of batch row s: ((first + s) * mul) mod n_data (a permutation
// of the data set when mul is coprime with n_data).
__device__ __forceinline__ long long sample_index(long long s, long long first, long long mul, long long n_data) {
    return (long long)(((unsigned long long)(first + s) % (unsigned long long)n_data) * (unsigned long long)mul %
                       (unsigned long long)n_data);
}

struct AdamArgs {
    float lr, beta1, beta2, eps, c1, c2;  // c1, c2: bias corrections 1/(1 - beta^t)
    int apply;                            // 0: gradients only
};

// bf16 / compact copies of one master weight.
__device__ __forceinline__ void mlp_refresh_one(const MlpDev& M, int p, float w) {
    if (p >= oW2 && p < ob2) {
        const int j = (p - oW2) / kMHid, k = (p - oW2) % kMHid;
        const __nv_bfloat16 b = __float2bfloat16_rn(w);
        M.W2b[j * kMHid + k] = b;
        M.W2Tb[k * kMHid + j] = b;
    } else if (p < ob1) {
        M.small[sW1 + p] = round_bf16(w);
    } else if (p < oW2) {
        M.small[sb1 + (p - ob1)] = w;
    } else if (p < oW3) {
        M.small[sb2 + (p - ob2)] = w;
    } else if (p < ob3) {
        M.small[sW3 + (p - oW3)] = round_bf16(w);
    } else {
        M.small[sb3 + (p - ob3)] = w;
    }
}

// x[0] + x[stride] + ... (n terms) added in this order, eight loads in flight.
__device__ __forceinline__ float ordered_sum(const float* x, int n, size_t stride) {
    float s = 0.f;
    int b = 0;
    for (; b + 8 <= n; b += 8) {
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = x[(size_t)(b + i) * stride];
#pragma unroll
        for (int i = 0; i < 8; ++i) s += v[i];
    }
    for (; b < n; ++b) s += x[(size_t)b * stride];
    return s;
}

// Sums the partials of n_part blocks in block order, writes the gradient and
// the batch loss (*loss), applies Adam to the masters and refreshes the rounded
// copies.
__global__ void k_mlp_update(MlpDev M, int n_part, int n_loss, float* loss, AdamArgs A) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p == kMParams) *loss = ordered_sum(M.loss_part, n_loss, 1);  // a thread past the parameters
    if (p >= kMParams) return;
    const float gsum = ordered_sum(M.grad_part + p, n_part, kMParams);
    M.grad[p] = gsum;
    if (!A.apply) return;
    const float m = A.beta1 * M.m[p] + (1.f - A.beta1) * gsum;
    const float v = A.beta2 * M.v[p] + (1.f - A.beta2) * gsum * gsum;
    M.m[p] = m;
    M.v[p] = v;
    const float w = M.master[p] - A.lr * (m * A.c1) / (sqrtf(v * A.c2) + A.eps);
    M.master[p] = w;
    mlp_refresh_one(M, p, w);
}

constexpr int kUpdateBlocks = (kMParams + 1 + 127) / 128;  // one thread per parameter and one for the loss

__global__ void k_mlp_refresh(MlpDev M) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < kMParams) mlp_refresh_one(M, p, M.master[p]);
}

// ------------------------------------------------------------ learned step

// Potential psi (psi' = E, psi(0) = 0) of the field the gather sees: E linear
// in each cell, so psi is quadratic there; off the mesh E = rE_edge / r.
__device__ __forceinline__ double psi_at(const LearnedArgs& A, double R) {
    if (A.field == PIC_FIELD_DUFFING) return -0.25 * ((R * R) * (R * R));
    if (A.field != PIC_FIELD_POISSON) return 0.0;
    const double x = (R - A.r_min) * A.inv_hr;
    if (x >= 0.0 && x < (double)A.n_cells) {
        const int j = (int)floor(x);
        const double d = R - (A.r_min + (double)j * A.hr);
        const double Ej = A.E[j], Ej1 = A.E[j + 1];
        return A.psi[j] + Ej * d + (Ej1 - Ej) * (d * d) * (0.5 * A.inv_hr);
    }
    if (x < 0.0) return A.psi[0] + A.edges[0] * log(R / A.r_min);
    return A.psi[A.n_cells] + A.edges[1] * log(R / -A.r_min);  // beyond r_max (NaN propagates)
}

// Frozen-field energy (R^2 + V^2)/2 - eps psi(R): conserved by the
// characteristics dR/dt = V/eps, dV/dt = -R/eps + E(R) when E does not change.
__device__ __forceinline__ double frozen_energy(const LearnedArgs& A, double R, double V) {
    return 0.5 * (R * R + V * V) - A.eps * psi_at(A, R);
}

// The FP64 rule, out of line: it runs only for the particles the binary32
// check leaves undecided (and for every particle of FP64 handles).
static __device__ __noinline__ bool frozen_keep_fp64(const LearnedArgs& A, double Rp, double Vp, double Rl,
                                                     double Vl) {
    const double H0 = frozen_energy(A, Rp, Vp);
    const double H1 = frozen_energy(A, Rl, Vl);
    return fabs(H1 - H0) <= A.tol * fabs(H0);
}

// ------------------------------------------------------------ tensor-core inference (tcgen05)
//
// Inference of the network (pic_mlp_forward) and the learned step's
// correction with the 64 x 64 hidden layer on the 5th-generation tensor
// cores: a block of 256 threads owns 128 samples, two threads each (warps 0..3
// the hidden units 0..31, warps 4..7 the others), writes bf16(gelu(z1)) as the
// A operand (128 x 64, K-major core matrices) to shared memory, and one thread
// issues four tcgen05.mma (M = 128, N = 64, K = 16 each) against W2 (B operand,
// 64 x 64) into a 64-column f32 accumulator in tensor memory and commits them
// to an mbarrier; each warp then reads half of its 32 rows back with
// tcgen05.ld.  The output layer adds the products of each sample's 64 columns
// in four fused multiply-add chains of 16 (columns 8 nt + 2 q + e for chain q)
// combined as (s0 + s1) + (s2 + s3); the first thread hands its chains to the
// second.  (Up to a few tiles per SM a call is one tile's latency: with one
// thread per sample, occupancy queries and a copy of the error flag on every
// call, 10^5 samples took 58 us and 100 samples 45, now 46 and 32; from 10^6 on,
// where issue binds, both take 0.17 us per 1000.)  Where a
// GELU is rounded to bfloat16 at once it is evaluated by gelu_for_bf16
// (gelu_fast.cuh), which rounds exactly as the erfc form does.

constexpr int kTcThreads = 128;  // samples of a tile (rows of the MMA)
constexpr int kInfThreads = 256; // two threads per sample
constexpr int kTcCols = 64;      // TMEM columns of the accumulator (N = 64, f32)

struct TcSmem {
    alignas(1024) unsigned char A[kTcThreads * kMHid * 2];  // bf16(h1): 128 x 64, K-major core matrices
    alignas(1024) unsigned char Bw[kMHid * kMHid * 2];      // W2: 64 (N) x 64 (K)
    float4 l1[kMHid][2];  // per hidden unit: (W1[j][0..3]), (W1[j][4], b1[j], 0, 0)
    float4 l3[kMHid];     // per hidden unit: (b2[j], W3[0][j], W3[1][j], 0)
    float b3[kMOut];
    float4 gtab[kGeluSeg + 1];  // segment table of gelu_for_bf16
    float4 acc[kMOut][kTcThreads];  // chains of the output layer, from a sample's first thread to its second
    unsigned long long mbar;
    unsigned int taddr;
    int fail;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 f32 columns [col, col + 16) of this warp's 32 TMEM lanes (lane = row of the tile)
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// mbarrier phase wait with a time limit; false when it ran out
__device__ __forceinline__ bool tc_wait(uint32_t mbar, uint32_t parity) {
    const long long t0 = clock64();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > (2ll << 30)) return false;  // ~1 s at 2 GHz
    }
}

// MODE 0: outputs to Y (pic_mlp_forward); 1, 2: the learned step's
// correction of an FP64 / FP32 state, kept where the frozen-field energy
// check allows it.
// Launch bounds for 3 / 4 / 6 blocks per SM, time of a learned binary32 step outside
// its window: 10^7 particles 2006 / 1855 / 1930 us (1990 with one thread per sample),
// 2 10^6 477 / 442 / 466 (532), 2 10^5 133 / 129 / 133 (208).  Six leave 40 registers and
// spill 52 bytes in MODE 2.
template <int MODE>
__global__ void __launch_bounds__(kInfThreads, 6) k_mlp_tc(MlpDev M, LearnedArgs A, const float* __restrict__ X,
                                                        float* __restrict__ Y, long long n) {
    __shared__ TcSmem S;
    extern __shared__ float s_tab[];  // binary32 field tables of the energy check (MODE 2, Poisson)
    const int t = threadIdx.x, warp = t >> 5;
    const int half = warp >> 2, row = t & (kTcThreads - 1);  // this thread's units 32 half .. + 31 of sample `row`
    // W2 as the B operand; the CUDA-core layers' weights packed per hidden unit
    for (int i = t; i < kMHid * kMHid / 8; i += kInfThreads) {
        const int nrow = i >> 3, kb = i & 7;  // 8 consecutive k of output row nrow
        *reinterpret_cast<uint4*>(S.Bw + tc_kmajor_offset(nrow, kb * 8)) =
            *reinterpret_cast<const uint4*>(M.W2b + nrow * kMHid + kb * 8);
    }
    if (t < kMHid) {
        const float* w1 = M.small + sW1 + t * kMIn;
        S.l1[t][0] = make_float4(w1[0], w1[1], w1[2], w1[3]);
        S.l1[t][1] = make_float4(w1[4], M.small[sb1 + t], 0.f, 0.f);
        S.l3[t] = make_float4(M.small[sb2 + t], M.small[sW3 + t], M.small[sW3 + kMHid + t], 0.f);
    }
    if (t < kMOut) S.b3[t] = M.small[sb3 + t];
    if (t <= kGeluSeg) S.gtab[t] = make_float4(c_gelu_tab[t][0], c_gelu_tab[t][1], c_gelu_tab[t][2], c_gelu_tab[t][3]);
    if (MODE == 2 && A.tab_f)
        for (int i = t; i < 3 * (A.n_cells + 1); i += kInfThreads) s_tab[i] = A.tab_f[i];
    if (t == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&S.mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        S.fail = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.taddr)),
                     "r"(kTcCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = S.taddr;
    const uint32_t idesc = tc_idesc_bf16_f32(kTcThreads, kMHid);
    const uint32_t a_base = smem_u32(S.A), b_base = smem_u32(S.Bw), mbar = smem_u32(&S.mbar);

    EnergyF32 E32;
    E32.field = A.field;
    E32.eps = (float)A.eps;
    E32.tol = (float)A.tol;
    E32.n_cells = A.n_cells;
    E32.r_min = (float)A.r_min;
    E32.hr = (float)A.hr;
    E32.inv_hr = (float)A.inv_hr;
    const float* tab_f = (MODE == 2 && A.tab_f) ? s_tab : nullptr;
    E32.E = tab_f;
    E32.slope = tab_f ? tab_f + (A.n_cells + 1) : nullptr;
    E32.psi = tab_f ? tab_f + 2 * (A.n_cells + 1) : nullptr;
    if (A.field == PIC_FIELD_POISSON && !tab_f) E32.field = -1;  // no tables: every particle in FP64

    unsigned int fallback = 0;
    uint32_t parity = 0;
    const long long tiles = (n + kTcThreads - 1) / kTcThreads;
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long long s = tile * kTcThreads + row;
        const bool valid = s < n;
        float x[kMIn];
        if (MODE == 0) {
#pragma unroll
            for (int i = 0; i < kMIn; ++i) x[i] = valid ? X[s * kMIn + i] : 0.f;
        } else {
            if (MODE == 1) {
                const double2 v = valid ? ((const double2*)A.y_prev)[s] : make_double2(0.0, 0.0);
                x[0] = (float)v.x;
                x[1] = (float)v.y;
            } else {
                const float2 v = valid ? ((const float2*)A.y_prev)[s] : make_float2(0.f, 0.f);
                x[0] = v.x;
                x[1] = v.y;
            }
            x[2] = A.in_sin;
            x[3] = A.in_cos;
            x[4] = A.in_dt;
        }
        // layer 1 + GELU into the A operand: row `row`, 8 columns (one 16-byte
        // core-matrix row) per pass; the pass loop stays rolled for the
        // instruction cache
#pragma unroll 1
        for (int kb = half * 4; kb < half * 4 + 4; ++kb) {
            unsigned int packed[4];
#pragma unroll
            for (int e = 0; e < 8; e += 2) {
                float h[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int col = kb * 8 + e + q;
                    const float4 wa = S.l1[col][0], wb = S.l1[col][1];
                    float z = wb.y;
                    z = fmaf(wa.x, x[0], z);
                    z = fmaf(wa.y, x[1], z);
                    z = fmaf(wa.z, x[2], z);
                    z = fmaf(wa.w, x[3], z);
                    z = fmaf(wb.x, x[4], z);
                    h[q] = gelu_for_bf16(z, S.gtab);  // rounded to bf16 by pack_bf16
                }
                packed[e >> 1] = pack_bf16(h[0], h[1]);
            }
            *reinterpret_cast<uint4*>(S.A + tc_kmajor_offset(row, kb * 8)) =
                make_uint4(packed[0], packed[1], packed[2], packed[3]);
        }
        // the generic-proxy writes of A become visible to the tensor core
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        if (t == 0) {
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < kMHid / 16; ++ks) {
                const uint64_t ad = tc_smem_desc(a_base + ks * 2 * kTcLbo, kTcLbo, kTcSbo);
                const uint64_t bd = tc_smem_desc(b_base + ks * 2 * kTcLbo, kTcLbo, kTcSbo);
                asm volatile(
                    "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(taddr),
                    "l"(ad), "l"(bd), "r"(idesc), "r"((uint32_t)ks)
                    : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                         : "memory");
        }
        if (!tc_wait(mbar, parity)) S.fail = 1;
        parity ^= 1u;
        tc_fence_after();
        __syncthreads();
        if (S.fail) break;
        // z2 = D + b2 of this thread's half row, GELU, bf16 (two per register)
        unsigned int h2[16];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float d[16];
            tc_ld16(taddr + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(half * 32 + c * 16), d);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int i = 0; i < 16; i += 2) {
                const int col = half * 32 + c * 16 + i;
                h2[c * 8 + (i >> 1)] = pack_bf16(gelu_for_bf16(d[i] + S.l3[col].x, S.gtab),
                                                 gelu_for_bf16(d[i + 1] + S.l3[col + 1].x, S.gtab));
            }
        }
        tc_fence_before();  // this tile's TMEM reads come before the next tile's MMA
        // output layer: the chains of columns 0..31, then of 32..63
        float acc[kMOut][4];
        if (half == 1) asm volatile("bar.sync 1, %0;" ::"n"(kInfThreads) : "memory");
#pragma unroll
        for (int o = 0; o < kMOut; ++o) {
            const float4 a = half ? S.acc[o][row] : make_float4(0.f, 0.f, 0.f, 0.f);
            acc[o][0] = a.x;
            acc[o][1] = a.y;
            acc[o][2] = a.z;
            acc[o][3] = a.w;
        }
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int q = (i & 7) >> 1;
            const float4 w = S.l3[half * 32 + i];
            const float h = __uint_as_float((i & 1) ? (h2[i >> 1] & 0xffff0000u) : (h2[i >> 1] << 16));
            acc[0][q] = fmaf(w.y, h, acc[0][q]);
            acc[1][q] = fmaf(w.z, h, acc[1][q]);
        }
        if (half == 0) {
#pragma unroll
            for (int o = 0; o < kMOut; ++o) S.acc[o][row] = make_float4(acc[o][0], acc[o][1], acc[o][2], acc[o][3]);
            // the second threads read the chains before the next tile's block barriers
            asm volatile("bar.arrive 1, %0;" ::"n"(kInfThreads) : "memory");
            continue;
        }
        float out[kMOut];
#pragma unroll
        for (int o = 0; o < kMOut; ++o) out[o] = ((acc[o][0] + acc[o][1]) + (acc[o][2] + acc[o][3])) + S.b3[o];
        if (!valid) continue;
        if (MODE == 0) {
            Y[s * kMOut] = out[0];
            Y[s * kMOut + 1] = out[1];
            continue;
        }
        const float dRf = A.scale_R * out[0], dVf = A.scale_V * out[1];
        if (dRf == 0.0f && dVf == 0.0f) continue;
        double Rp, Vp, Rl, Vl;
        int dec = -1;
        if (MODE == 1) {
            const double2 pl = ((const double2*)A.y)[s];
            Rp = pl.x;
            Vp = pl.y;
            Rl = pl.x + (double)dRf;
            Vl = pl.y + (double)dVf;
        } else {
            const float2 pl = ((const float2*)A.y)[s];
            const float R1 = pl.x + dRf, V1 = pl.y + dVf;
            Rp = pl.x;
            Vp = pl.y;
            Rl = (double)R1;
            Vl = (double)V1;
            // binary32 where it provably gives the FP64 decision
            dec = energy_check_f32(E32, pl.x, pl.y, R1, V1);
        }
        // the plain step judges: the correction may move the frozen-field
        // energy away from the plain step's by at most tol |H|
        const bool keep = dec >= 0 ? dec == 1 : frozen_keep_fp64(A, Rp, Vp, Rl, Vl);
        if (keep) {
            if (MODE == 1) ((double2*)A.y)[s] = make_double2(Rl, Vl);
            else ((float2*)A.y)[s] = make_float2((float)Rl, (float)Vl);
        } else {
            ++fallback;
        }
    }
    if (MODE != 0) {
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) fallback += __shfl_xor_sync(0xffffffffu, fallback, d);
        if ((t & 31) == 0 && fallback) atomicAdd(A.n_fallback, (unsigned long long)fallback);
    }
    if (t == 0 && S.fail) *(volatile int*)M.err = 1;
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(kTcCols) : "memory");
    }
}

// Blocks of k_mlp_tc resident on one SM, from its registers, its shared
// memory and its 64 tensor-memory columns (512 per SM).  The runtime's
// occupancy query answers 1 for this kernel, which would leave 7 of every 8
// warp slots it could use empty.
static int tc_blocks_per_sm(const void* fn, size_t dyn_smem) {
    cudaFuncAttributes fa;
    int dev = 0, smem_sm = 0, resv = 0, regs_sm = 0;
    if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&resv, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess)
        return 1;
    const int regs_block = ((fa.numRegs + 7) / 8) * 8 * kInfThreads;  // allocated per warp in units of 8 per thread
    int k = 512 / kTcCols;
    k = std::min(k, 2048 / kInfThreads);
    if (regs_block > 0) k = std::min(k, regs_sm / regs_block);
    k = std::min(k, (int)((size_t)smem_sm / (fa.sharedSizeBytes + dyn_smem + (size_t)resv)));
    return k < 1 ? 1 : k;
}

static void* tc_fn(int mode) {
    return mode == 0 ? (void*)k_mlp_tc<0> : mode == 1 ? (void*)k_mlp_tc<1> : (void*)k_mlp_tc<2>;
}
// Sets up the inference kernel of a mode for its dynamic shared memory and
// returns the blocks resident per SM.
static cudaError_t tc_setup(int mode, size_t smem, int* per_sm) {
    cudaError_t e = cudaFuncSetAttribute(tc_fn(mode), cudaFuncAttributePreferredSharedMemoryCarveout,
                                         (int)cudaSharedmemCarveoutMaxShared);
    // 48 KB without opting in hold the kernel's own arrays and the energy check's
    // tables together: 33 KB leave room for 1278 cells
    if (e == cudaSuccess && smem > 0) e = open_shared_memory(tc_fn(mode), nullptr);
    if (e == cudaSuccess) *per_sm = tc_blocks_per_sm(tc_fn(mode), smem);
    return e;
}

// Launch of the tensor-core inference over n samples: as many blocks as are
// resident at once (per_sm each, as tc_setup gave), no more blocks than tiles.
static cudaError_t launch_mlp_tc(const MlpDev& D, const LearnedArgs& A, int mode, const float* X, float* Y, long long n,
                                 size_t smem, int per_sm, int sm_count, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const long long tiles = (n + kTcThreads - 1) / kTcThreads;
    const long long cap = (long long)sm_count * per_sm;
    const int grid = (int)(tiles < cap ? tiles : cap);
    if (mode == 0) k_mlp_tc<0><<<grid, kInfThreads, smem, st>>>(D, A, X, Y, n);
    else if (mode == 1) k_mlp_tc<1><<<grid, kInfThreads, smem, st>>>(D, A, X, Y, n);
    else k_mlp_tc<2><<<grid, kInfThreads, smem, st>>>(D, A, X, Y, n);
    return cudaGetLastError();
}

// ------------------------------------------------------------ tensor-core training (tcgen05)
//
// One block of 512 threads per tile of 128 samples: warp w works on the
// samples (tensor-memory lanes) 32 (w mod 4) .. + 31 and the hidden units
// 16 (w / 4) .. + 15, so a sample's units are spread over four warps.
//   z1, h1                      -> A operand, and transposed for the gradients
//   MMA 1: z2 = bf16(h1) W2^T   (then + b2), h2, the output layer: its four
//                               chains (the order of k_mlp_tc) pass through the
//                               four warps of a sample in turn
//   dz2 = (dout W3) gelu'(z2)   -> A operand, and transposed
//   MMA 2: dh1 = bf16(dz2) W2;  MMA 3: dW2 += bf16(dz2)^T h1 over the tile's
//                               samples, kept in tensor memory over the block's
//                               tiles (rows 64..127 of the operand are zero)
//   dz1 = dh1 gelu'(z1)
//   dW1, db1, db2, dW3, db3     on the CUDA cores, sums over the tile in registers
// Rows past the batch enter every sum as zeros, whatever the weights (an
// infinite weight times a zero dout would be NaN).
// Nothing per sample goes through global memory.  The step is latency-bound
// (64 tiles at the usual batch of 8192): with one thread per sample and a
// second kernel that reloaded every record for the gradients, the two took 32
// and 20 us and a third and fourth summed and refreshed in 11; now it is 23.5
// and 4.9 us, without the wait for every loss: 5 steps and a gradient 551 -> 301 us.
// Beyond 152 tiles a block of an SM takes several: the same calls with a batch of
// 4 10^4 896 -> 493 us, 2 10^5 2.81 -> 1.19 ms, 10^6 11.2 -> 4.75 ms.

constexpr int kTrThreads = 512;
constexpr int kTrRow = kMHid + 4;    // floats per row: 16-byte rows that start 4 banks apart
constexpr int kTrRowB = kMHid + 8;   // bf16 per row, the same
constexpr int kTrParts = kTrThreads / kMHid;
constexpr int kTrSums = 9;           // dW1 (5), db1, db2, dW3 (2) of one hidden unit

struct TcTrainSmem {
    alignas(1024) unsigned char A[kTcThreads * kMHid * 2];      // bf16(h1), then bf16(dz2): 128 x 64, K-major
    alignas(1024) unsigned char At[2][kTcThreads * kMHid * 2];  // bf16(dz2)^T: 64 (of 128) units x 64 samples, both halves
    alignas(1024) unsigned char Bw[kMHid * kMHid * 2];          // W2: N = j, K = k
    alignas(1024) unsigned char Bt[kMHid * kMHid * 2];          // W2^T: N = k, K = j
    alignas(1024) unsigned char Ht[2][kMHid * kMHid * 2];       // bf16(h1)^T: 64 units x 64 samples, both halves
    float d1[kTcThreads][kTrRow];             // z1, then gelu'(z1), then dz1
    float d2[kTcThreads][kTrRow];             // z2, then dz2
    __nv_bfloat16 h2[kTcThreads][kTrRowB];
    float4 xd[kTcThreads][2];                 // x, dout
    float4 acc[kTcThreads][kMOut];            // chains of the output layer between warps
    float4 l1[kMHid][2];
    float4 l3[kMHid];
    float b3[kMOut];
    float4 gtab[kGeluSeg + 1];
    unsigned long long mbar;
    unsigned int taddr;
    int fail;
    float loss[kTcThreads / 32];
};

// Thread 0: the four K = 16 MMAs of a K = 64 product into the accumulator at
// taddr (accumulating onto it when acc).
__device__ __forceinline__ void tc_issue_k64(uint32_t taddr, uint32_t a_base, uint32_t b_base, uint32_t idesc,
                                             bool acc) {
#pragma unroll
    for (int ks = 0; ks < kMHid / 16; ++ks) {
        const uint64_t ad = tc_smem_desc(a_base + ks * 2 * kTcLbo, kTcLbo, kTcSbo);
        const uint64_t bd = tc_smem_desc(b_base + ks * 2 * kTcLbo, kTcLbo, kTcSbo);
        const uint32_t en = (acc || ks > 0) ? 1u : 0u;
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(taddr),
            "l"(ad), "l"(bd), "r"(idesc), "r"(en)
            : "memory");
    }
}
__device__ __forceinline__ void tc_commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

// A 64 x 64 bf16 matrix (row-major, rows along N) as a K-major B operand.
__device__ __forceinline__ void tc_stage_b(unsigned char* dst, const __nv_bfloat16* __restrict__ src) {
    for (int i = threadIdx.x; i < kMHid * kMHid / 8; i += blockDim.x) {
        const int nrow = i >> 3, kb = i & 7;
        *reinterpret_cast<uint4*>(dst + tc_kmajor_offset(nrow, kb * 8)) =
            *reinterpret_cast<const uint4*>(src + nrow * kMHid + kb * 8);
    }
}

// Every thread's operand writes become visible to the tensor core behind the
// block barrier.
__device__ __forceinline__ void tc_operands_ready() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
}
// Every thread waits for the committed MMAs; false (and the block's fail flag)
// when the wait ran out of time.
__device__ __forceinline__ bool tc_block_wait(uint32_t mbar, uint32_t& parity, int& fail) {
    if (!tc_wait(mbar, parity)) fail = 1;
    parity ^= 1u;
    tc_fence_after();
    __syncthreads();
    return !fail;
}

// Four consecutive units of one row of an operand and of its transpose.
__device__ __forceinline__ void tc_put4(unsigned char* A, unsigned char* T, int row, int col, const float (&v)[4]) {
    const unsigned int lo = pack_bf16(v[0], v[1]), hi = pack_bf16(v[2], v[3]);
    *reinterpret_cast<uint2*>(A + tc_kmajor_offset(row, col)) = make_uint2(lo, hi);
    const int k = row & (kMHid - 1);
    *reinterpret_cast<unsigned short*>(T + tc_kmajor_offset(col, k)) = (unsigned short)lo;
    *reinterpret_cast<unsigned short*>(T + tc_kmajor_offset(col + 1, k)) = (unsigned short)(lo >> 16);
    *reinterpret_cast<unsigned short*>(T + tc_kmajor_offset(col + 2, k)) = (unsigned short)hi;
    *reinterpret_cast<unsigned short*>(T + tc_kmajor_offset(col + 3, k)) = (unsigned short)(hi >> 16);
}

__global__ void __launch_bounds__(kTrThreads) k_mlp_train_tc(MlpDev M, const float* __restrict__ X,
                                                             const float* __restrict__ Y, long long B, long long first,
                                                             long long mul, long long n_data, float invB) {
    extern __shared__ __align__(1024) unsigned char train_smem[];
    TcTrainSmem& S = *reinterpret_cast<TcTrainSmem*>(train_smem);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int cb = warp >> 2, row = (warp & 3) * 32 + lane;  // this thread's units 16 cb .. + 15 of sample `row`
    tc_stage_b(S.Bw, M.W2b);
    tc_stage_b(S.Bt, M.W2Tb);
    for (int i = t; i < (int)(sizeof(S.At) / 16); i += kTrThreads)
        reinterpret_cast<uint4*>(S.At)[i] = make_uint4(0, 0, 0, 0);
    if (t < kMHid) {
        const float* w1 = M.small + sW1 + t * kMIn;
        S.l1[t][0] = make_float4(w1[0], w1[1], w1[2], w1[3]);
        S.l1[t][1] = make_float4(w1[4], M.small[sb1 + t], 0.f, 0.f);
        S.l3[t] = make_float4(M.small[sb2 + t], M.small[sW3 + t], M.small[sW3 + kMHid + t], 0.f);
    }
    if (t < kMOut) S.b3[t] = M.small[sb3 + t];
    if (t <= kGeluSeg) S.gtab[t] = make_float4(c_gelu_tab[t][0], c_gelu_tab[t][1], c_gelu_tab[t][2], c_gelu_tab[t][3]);
    if (t == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&S.mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        S.fail = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.taddr)),
                     "r"(2 * kTcCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // columns 0..63: z2, then dh1; columns 64..127: dW2
    const uint32_t taddr = S.taddr, tgrad = taddr + kTcCols;
    const uint32_t lane0 = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t idesc = tc_idesc_bf16_f32(kTcThreads, kMHid);
    const uint32_t a_base = smem_u32(S.A), mbar = smem_u32(&S.mbar);
    unsigned char* const Atr = S.At[row >> 6];
    unsigned char* const Htr = S.Ht[row >> 6];
    uint32_t parity = 0;
    float loss = 0.f;
    float gs[kTrSums], gb3[kMOut] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < kTrSums; ++i) gs[i] = 0.f;
    bool any = false;
    const long long tiles = (B + kTcThreads - 1) / kTcThreads;
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long long s = tile * kTcThreads + row;
        const bool valid = s < B;
        const long long idx = valid ? sample_index(s, first, mul, n_data) : 0;
        float x[kMIn];
#pragma unroll
        for (int i = 0; i < kMIn; ++i) x[i] = valid ? X[idx * kMIn + i] : 0.f;
        // layer 1 + GELU
#pragma unroll 1
        for (int c = cb * 16; c < cb * 16 + 16; c += 4) {
            float z[4], h[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 wa = S.l1[c + q][0], wb = S.l1[c + q][1];
                z[q] = wb.y;
                z[q] = fmaf(wa.x, x[0], z[q]);
                z[q] = fmaf(wa.y, x[1], z[q]);
                z[q] = fmaf(wa.z, x[2], z[q]);
                z[q] = fmaf(wa.w, x[3], z[q]);
                z[q] = fmaf(wb.x, x[4], z[q]);
                h[q] = valid ? gelu_for_bf16(z[q], S.gtab) : 0.f;
            }
            *reinterpret_cast<float4*>(&S.d1[row][c]) = make_float4(z[0], z[1], z[2], z[3]);
            tc_put4(S.A, Htr, row, c, h);
        }
        tc_operands_ready();
        if (t == 0) {
            tc_fence_after();
            tc_issue_k64(taddr, a_base, smem_u32(S.Bw), idesc, false);
            tc_commit(mbar);
        }
        if (!tc_block_wait(mbar, parity, S.fail)) break;
        {
            float d[16];
            tc_ld16(taddr + lane0 + (uint32_t)(cb * 16), d);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int i = 0; i < 16; i += 4)
                *reinterpret_cast<float4*>(&S.d2[row][cb * 16 + i]) =
                    make_float4(d[i] + S.l3[cb * 16 + i].x, d[i + 1] + S.l3[cb * 16 + i + 1].x,
                                d[i + 2] + S.l3[cb * 16 + i + 2].x, d[i + 3] + S.l3[cb * 16 + i + 3].x);
        }
#pragma unroll 1
        for (int c = cb * 16; c < cb * 16 + 16; c += 4) {
            const float4 z = *reinterpret_cast<const float4*>(&S.d2[row][c]);
            const uint2 h = make_uint2(pack_bf16(gelu_for_bf16(z.x, S.gtab), gelu_for_bf16(z.y, S.gtab)),
                                       pack_bf16(gelu_for_bf16(z.z, S.gtab), gelu_for_bf16(z.w, S.gtab)));
            *reinterpret_cast<uint2*>(&S.h2[row][c]) = valid ? h : make_uint2(0u, 0u);
        }
        // output layer: chain q takes the columns 8 nt + 2 q + e in order, warp by warp
#pragma unroll 1
        for (int g = 0; g < 4; ++g) {
            if (cb == g) {
                float acc[kMOut][4];
#pragma unroll
                for (int o = 0; o < kMOut; ++o) {
                    const float4 a = g ? S.acc[row][o] : make_float4(0.f, 0.f, 0.f, 0.f);
                    acc[o][0] = a.x;
                    acc[o][1] = a.y;
                    acc[o][2] = a.z;
                    acc[o][3] = a.w;
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const int q = (i & 7) >> 1;
                    const float4 w = S.l3[g * 16 + i];
                    const float h = __bfloat162float(S.h2[row][g * 16 + i]);
                    acc[0][q] = fmaf(w.y, h, acc[0][q]);
                    acc[1][q] = fmaf(w.z, h, acc[1][q]);
                }
                if (g < 3) {
#pragma unroll
                    for (int o = 0; o < kMOut; ++o)
                        S.acc[row][o] = make_float4(acc[o][0], acc[o][1], acc[o][2], acc[o][3]);
                } else {
                    float dout[kMOut];
#pragma unroll
                    for (int o = 0; o < kMOut; ++o) {
                        const float out = ((acc[o][0] + acc[o][1]) + (acc[o][2] + acc[o][3])) + S.b3[o];
                        const float d = valid ? out - Y[idx * kMOut + o] : 0.f;
                        loss = fmaf(d, d, loss);
                        dout[o] = d * invB;
                    }
                    S.xd[row][0] = make_float4(x[0], x[1], x[2], x[3]);
                    S.xd[row][1] = make_float4(x[4], dout[0], dout[1], 0.f);
                }
            }
            __syncthreads();
        }
        // dz2 = (dout W3) gelu'(z2)
        const float4 xd1 = S.xd[row][1];
#pragma unroll 1
        for (int c = cb * 16; c < cb * 16 + 16; c += 4) {
            float4* zp = reinterpret_cast<float4*>(&S.d2[row][c]);
            const float4 z4 = *zp;
            float v[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 w = S.l3[c + q];
                v[q] = valid ? fmaf(w.z, xd1.z, w.y * xd1.y) * gelu_d(v[q]) : 0.f;
            }
            *zp = make_float4(v[0], v[1], v[2], v[3]);
            tc_put4(S.A, Atr, row, c, v);
        }
        tc_operands_ready();
        if (t == 0) {
            tc_fence_after();
            tc_issue_k64(taddr, a_base, smem_u32(S.Bt), idesc, false);
            tc_issue_k64(tgrad, smem_u32(S.At[0]), smem_u32(S.Ht[0]), idesc, any);
            tc_issue_k64(tgrad, smem_u32(S.At[1]), smem_u32(S.Ht[1]), idesc, true);
            tc_commit(mbar);
        }
        any = true;
        // gelu'(z1) while the products run
#pragma unroll 1
        for (int c = cb * 16; c < cb * 16 + 16; c += 4) {
            float4* zp = reinterpret_cast<float4*>(&S.d1[row][c]);
            const float4 z = *zp;
            *zp = make_float4(gelu_d(z.x), gelu_d(z.y), gelu_d(z.z), gelu_d(z.w));
        }
        if (!tc_block_wait(mbar, parity, S.fail)) break;
        {
            float d[16];
            tc_ld16(taddr + lane0 + (uint32_t)(cb * 16), d);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int i = 0; i < 16; i += 4) {
                float4* gp = reinterpret_cast<float4*>(&S.d1[row][cb * 16 + i]);
                const float4 g = *gp;
                *gp = valid ? make_float4(d[i] * g.x, d[i + 1] * g.y, d[i + 2] * g.z, d[i + 3] * g.w)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        tc_fence_before();  // this tile's TMEM reads come before the next tile's MMA
        __syncthreads();
        // the small gradients: unit j, sixteen samples per thread
        const int j = t & (kMHid - 1), s0 = (t / kMHid) * (kTcThreads / kTrParts);
#pragma unroll 4
        for (int q = s0; q < s0 + kTcThreads / kTrParts; ++q) {
            const float4 xa = S.xd[q][0], xb = S.xd[q][1];
            const float d1 = S.d1[q][j], d2 = S.d2[q][j], h = __bfloat162float(S.h2[q][j]);
            gs[0] = fmaf(d1, xa.x, gs[0]);
            gs[1] = fmaf(d1, xa.y, gs[1]);
            gs[2] = fmaf(d1, xa.z, gs[2]);
            gs[3] = fmaf(d1, xa.w, gs[3]);
            gs[4] = fmaf(d1, xb.x, gs[4]);
            gs[5] += d1;
            gs[6] += d2;
            gs[7] = fmaf(xb.y, h, gs[7]);
            gs[8] = fmaf(xb.z, h, gs[8]);
            gb3[0] += xb.y;
            gb3[1] += xb.z;
        }
        __syncthreads();  // the next tile overwrites the rows
    }
    // partials of this block: the loss (fixed reduction order) ...
    if (cb == 3) {
#pragma unroll
        for (int dd = 16; dd >= 1; dd >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, dd);
        if (lane == 0) S.loss[warp & 3] = loss;
    }
    // ... the small gradients, summed over the parts in order ...
    __syncthreads();
    constexpr int kSumRow = kTrSums + kMOut;
    float* sums = &S.d1[0][0];  // [part][unit][kSumRow]
    static_assert(kTrParts * kMHid * kSumRow <= kTcThreads * kTrRow, "the partial sums fit the rows");
    {
        float* mine = sums + (size_t)t * kSumRow;
#pragma unroll
        for (int i = 0; i < kTrSums; ++i) mine[i] = gs[i];
        mine[kTrSums] = gb3[0];
        mine[kTrSums + 1] = gb3[1];
    }
    __syncthreads();
    float* part = M.grad_part + (size_t)blockIdx.x * kMParams;
    for (int i = t; i < kMHid * kSumRow; i += kTrThreads) {
        const int unit = i / kSumRow, q = i % kSumRow;
        float v = 0.f;
#pragma unroll
        for (int p = 0; p < kTrParts; ++p) v += sums[((size_t)p * kMHid + unit) * kSumRow + q];
        if (q < kMIn) part[oW1 + unit * kMIn + q] = v;
        else if (q == 5) part[ob1 + unit] = v;
        else if (q == 6) part[ob2 + unit] = v;
        else if (q < kTrSums) part[oW3 + (q - 7) * kMHid + unit] = v;
        else if (unit == 0) part[ob3 + (q - kTrSums)] = v;
    }
    // ... and dW2: accumulator lanes 0..63 are the rows j
    if (row < kMHid) {
        float d[16];
        tc_ld16(tgrad + lane0 + (uint32_t)(cb * 16), d);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int i = 0; i < 16; ++i) part[oW2 + row * kMHid + cb * 16 + i] = any && !S.fail ? d[i] : 0.f;
    }
    if (t == 0) {
        float sum = 0.f;
        for (int i = 0; i < kTcThreads / 32; ++i) sum += S.loss[i];
        M.loss_part[blockIdx.x] = 0.5f * sum * invB;
        if (S.fail) *(volatile int*)M.err = 1;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(2 * kTcCols) : "memory");
    }
}

// psi_c = 0 at the centre and psi_j the trapezoid sums outward, one half of the
// block for each side: every thread sums a run of cells, the runs are scanned
// (warp shuffles, then the warps' totals), and the thread walks its run again.
// A single thread's chain of 512 dependent FP64 additions took 68 us; the scan
// also adds in fewer roundings.
constexpr int kPsiThreads = 1024;
__global__ void __launch_bounds__(kPsiThreads) k_psi_nodes(const double* __restrict__ E, int n_cells, double hr,
                                                           double* __restrict__ psi, float* __restrict__ tab_f) {
    constexpr int H = kPsiThreads / 2;
    __shared__ double s_tot[kPsiThreads / 32];
    const int c = n_cells / 2, left = threadIdx.x >= H ? 1 : 0, t = threadIdx.x - left * H;
    const int lane = threadIdx.x & 31, w = t >> 5;
    const int cells = left ? c : n_cells - c, per = (cells + H - 1) / H;
    const int beg = min(t * per, cells), end = min(beg + per, cells);
    // cell k of a side lies between nodes c + d k and c + d (k + 1)
    const int d = left ? -1 : 1;
    auto inc = [&](int k) -> double { return (0.5 * hr) * (E[c + d * k] + E[c + d * (k + 1)]); };
    double sum = 0.0;
    for (int k = beg; k < end; ++k) sum += inc(k);
    double x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_tot[threadIdx.x >> 5] = x;
    __syncthreads();
    double run = __shfl_up_sync(0xffffffffu, x, 1);
    if (lane == 0) run = 0.0;
    double before = 0.0;
    for (int v = 0; v < w; ++v) before += s_tot[left * (H / 32) + v];
    run += before;
    if (threadIdx.x == 0) psi[c] = 0.0;
    for (int k = beg; k < end; ++k) {
        run += inc(k);
        psi[c + d * (k + 1)] = left ? -run : run;
    }
    if (!tab_f) return;
    __syncthreads();
    // binary32 copies for the energy check of the FP32 form
    const int Np1 = n_cells + 1;
    const double inv_hr = 1.0 / hr;
    for (int j = threadIdx.x; j < Np1; j += blockDim.x) {
        tab_f[j] = (float)E[j];
        tab_f[Np1 + j] = j < n_cells ? (float)((E[j + 1] - E[j]) * inv_hr) : 0.0f;
        tab_f[2 * Np1 + j] = (float)psi[j];
    }
}

cudaError_t launch_psi_nodes(const double* E, int n_cells, double hr, double* psi, cudaStream_t st,
                             long long* launches, float* tab_f) {
    k_psi_nodes<<<1, kPsiThreads, 0, st>>>(E, n_cells, hr, psi, tab_f);
    if (launches) ++*launches;
    return cudaGetLastError();
}

// psi at n positions: the same psi_at the learned step's FP64 energy check uses.
__global__ void k_psi_eval(LearnedArgs A, const double* __restrict__ R, double* __restrict__ out) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < A.n; i += stride) out[i] = psi_at(A, R[i]);
}

cudaError_t launch_psi_eval(const LearnedArgs& A, const double* R, double* out, int sm_count, cudaStream_t st) {
    if (A.n == 0) return cudaSuccess;
    const long long want = (A.n + 255) / 256;
    const int grid = (int)(want < (long long)sm_count * 4 ? want : (long long)sm_count * 4);
    k_psi_eval<<<grid, 256, 0, st>>>(A, R, out);
    return cudaGetLastError();
}

}  // namespace pic

// ------------------------------------------------------------ C ABI

struct pic_mlp {
    pic::MlpDev D;
    long long max_batch = 0;
    cudaStream_t st = nullptr;
    int sm_count = 0;
    long long t = 0;  // Adam steps taken
    int forward_per_sm = 1;  // resident blocks of the inference kernel (pic_mlp_forward) per SM
    int* err_host = nullptr;  // D.err as the host sees it
    std::vector<void*> allocs;
};

namespace {

int mlp_map(cudaError_t e) {
    if (e == cudaSuccess) return PIC_OK;
    if (e == cudaErrorMemoryAllocation) return PIC_ERR_NO_MEMORY;
    return PIC_ERR_CUDA;
}

template <typename T>
cudaError_t mlp_alloc(pic_mlp* m, T** p, size_t count) {
    void* q = nullptr;
    cudaError_t e = cudaMalloc(&q, sizeof(T) * (count ? count : 1));
    if (e == cudaSuccess) m->allocs.push_back(q);
    *p = (T*)q;
    return e;
}

void mlp_free(pic_mlp* m) {
    for (void* p : m->allocs) cudaFree(p);
    m->allocs.clear();
    if (m->err_host) cudaFreeHost(m->err_host);
    m->err_host = nullptr;
}

// Forward, backward and gradients, then their sum (+ Adam when apply); the
// batch loss goes to *loss (device).
cudaError_t mlp_step(pic_mlp* m, long long B, const float* X, const float* Y, long long first, long long mul,
                     long long n_data, float* loss, int apply, const pic_adam_t* opt) {
    pic::MlpDev& D = m->D;
    const long long tiles = (B + pic::kTcThreads - 1) / pic::kTcThreads;
    const int grid = (int)(tiles < m->sm_count ? tiles : m->sm_count);  // one block per SM (its shared memory)
    pic::k_mlp_train_tc<<<grid, pic::kTrThreads, sizeof(pic::TcTrainSmem), m->st>>>(D, X, Y, B, first, mul, n_data,
                                                                                   1.0f / (float)B);
    pic::AdamArgs A;
    std::memset(&A, 0, sizeof(A));
    if (apply) {
        m->t += 1;
        A.lr = opt->lr;
        A.beta1 = opt->beta1;
        A.beta2 = opt->beta2;
        A.eps = opt->eps;
        A.c1 = (float)(1.0 / (1.0 - std::pow((double)opt->beta1, (double)m->t)));
        A.c2 = (float)(1.0 / (1.0 - std::pow((double)opt->beta2, (double)m->t)));
        A.apply = 1;
    }
    pic::k_mlp_update<<<pic::kUpdateBlocks, 128, 0, m->st>>>(D, grid, grid, loss, A);
    return cudaGetLastError();
}

long long gcd_ll(long long a, long long b) {
    while (b) {
        const long long r = a % b;
        a = b;
        b = r;
    }
    return a;
}

}  // namespace

namespace pic {
cudaError_t launch_learned_apply(const pic_mlp* m, const LearnedArgs& A, int sm_count, cudaStream_t st,
                                 long long* launches) {
    if (A.n == 0) return cudaSuccess;
    const int mode = A.prec == 0 ? 1 : 2;
    const size_t smem = (mode == 2 && A.tab_f) ? sizeof(float) * 3 * (size_t)(A.n_cells + 1) : 0;
    int per_sm = 1;
    cudaError_t e = tc_setup(mode, smem, &per_sm);
    if (e == cudaSuccess) e = launch_mlp_tc(m->D, A, mode, nullptr, nullptr, A.n, smem, per_sm, sm_count, st);
    if (launches) ++*launches;
    return e;
}

// PIC_ERR_TIMEOUT (and the flag cleared) when a tensor-core wait of the
// inference kernel ran out of time since the last call; synchronises st.
int mlp_take_error(const pic_mlp* m, cudaStream_t st) {
    const cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? PIC_ERR_NO_MEMORY : PIC_ERR_CUDA;
    volatile int* err = m->err_host;
    if (!*err) return PIC_OK;
    *err = 0;
    return PIC_ERR_TIMEOUT;
}
}  // namespace pic

extern "C" {

int pic_mlp_num_params(void) { return pic::kMParams; }

int pic_mlp_create(int64_t max_batch, void* stream, pic_mlp** out) {
    if (!out || max_batch < 1 || max_batch > (1ll << 26)) return PIC_ERR_INVALID_ARG;
    *out = nullptr;
    int dev = 0, sms = 0, count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || count == 0) return PIC_ERR_CUDA;
    if (cudaGetDevice(&dev) != cudaSuccess) return PIC_ERR_CUDA;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return PIC_ERR_CUDA;
    pic_mlp* m = new (std::nothrow) pic_mlp();
    if (!m) return PIC_ERR_NO_MEMORY;
    m->max_batch = max_batch;
    m->st = (cudaStream_t)stream;
    m->sm_count = sms;
    pic::MlpDev& D = m->D;
    std::memset(&D, 0, sizeof(D));
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess) e = mlp_alloc(m, &D.master, pic::kMParams);
    if (e == cudaSuccess) e = mlp_alloc(m, &D.m, pic::kMParams);
    if (e == cudaSuccess) e = mlp_alloc(m, &D.v, pic::kMParams);
    if (e == cudaSuccess) e = mlp_alloc(m, &D.W2b, pic::kMHid * pic::kMHid);
    if (e == cudaSuccess) e = mlp_alloc(m, &D.W2Tb, pic::kMHid * pic::kMHid);
    if (e == cudaSuccess) e = mlp_alloc(m, &D.small, pic::kMSmall);
    if (e == cudaSuccess) e = mlp_alloc(m, &D.loss_part, (size_t)sms);
    if (e == cudaSuccess) e = mlp_alloc(m, &D.grad_part, (size_t)sms * pic::kMParams);
    if (e == cudaSuccess) e = mlp_alloc(m, &D.grad, pic::kMParams);
    if (e == cudaSuccess) e = mlp_alloc(m, &D.loss, pic::kLossHist);
    if (e == cudaSuccess) e = cudaHostAlloc((void**)&m->err_host, sizeof(int), cudaHostAllocMapped);
    if (e == cudaSuccess) *m->err_host = 0;
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void**)&D.err, m->err_host, 0);
    if (e == cudaSuccess) e = pic::tc_setup(0, 0, &m->forward_per_sm);
    if (e == cudaSuccess) e = cudaMemsetAsync(D.master, 0, sizeof(float) * pic::kMParams, m->st);
    if (e == cudaSuccess) e = cudaMemsetAsync(D.m, 0, sizeof(float) * pic::kMParams, m->st);
    if (e == cudaSuccess) e = cudaMemsetAsync(D.v, 0, sizeof(float) * pic::kMParams, m->st);
    if (e == cudaSuccess) {
        pic::k_mlp_refresh<<<(pic::kMParams + 255) / 256, 256, 0, m->st>>>(D);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(pic::k_mlp_train_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(pic::TcTrainSmem));
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->st);
    if (e != cudaSuccess) {
        mlp_free(m);
        delete m;
        return mlp_map(e);
    }
    *out = m;
    return PIC_OK;
}

int pic_mlp_set_weights(pic_mlp* m, const float* w, int ptr_kind) {
    if (!m || !w || (ptr_kind != PIC_PTR_HOST && ptr_kind != PIC_PTR_DEVICE)) return PIC_ERR_INVALID_ARG;
    cudaError_t e = cudaMemcpyAsync(m->D.master, w, sizeof(float) * pic::kMParams,
                                    ptr_kind == PIC_PTR_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, m->st);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->D.m, 0, sizeof(float) * pic::kMParams, m->st);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->D.v, 0, sizeof(float) * pic::kMParams, m->st);
    if (e == cudaSuccess) {
        pic::k_mlp_refresh<<<(pic::kMParams + 255) / 256, 256, 0, m->st>>>(m->D);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->st);
    m->t = 0;
    return mlp_map(e);
}

int pic_mlp_get_weights(pic_mlp* m, float* w, int ptr_kind) {
    if (!m || !w || (ptr_kind != PIC_PTR_HOST && ptr_kind != PIC_PTR_DEVICE)) return PIC_ERR_INVALID_ARG;
    cudaError_t e = cudaMemcpyAsync(w, m->D.master, sizeof(float) * pic::kMParams,
                                    ptr_kind == PIC_PTR_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, m->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->st);
    return mlp_map(e);
}

int pic_mlp_forward(pic_mlp* m, int64_t n, const float* X_dev, float* Y_dev) {
    if (!m || n < 0 || (n > 0 && (!X_dev || !Y_dev))) return PIC_ERR_INVALID_ARG;
    if (n == 0) return PIC_OK;
    pic::LearnedArgs A;
    std::memset(&A, 0, sizeof(A));
    const cudaError_t e = pic::launch_mlp_tc(m->D, A, 0, X_dev, Y_dev, n, 0, m->forward_per_sm, m->sm_count, m->st);
    if (e != cudaSuccess) return mlp_map(e);
    return pic::mlp_take_error(m, m->st);
}

int pic_mlp_gradients(pic_mlp* m, int64_t n, const float* X_dev, const float* T_dev, float* grad, float* loss,
                      int ptr_kind) {
    if (!m || n < 1 || n > m->max_batch || !X_dev || !T_dev || !grad || !loss) return PIC_ERR_INVALID_ARG;
    if (ptr_kind != PIC_PTR_HOST && ptr_kind != PIC_PTR_DEVICE) return PIC_ERR_INVALID_ARG;
    const cudaMemcpyKind k = ptr_kind == PIC_PTR_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    cudaError_t e = mlp_step(m, n, X_dev, T_dev, 0, 1, n, m->D.loss, 0, nullptr);
    if (e == cudaSuccess) e = cudaMemcpyAsync(grad, m->D.grad, sizeof(float) * pic::kMParams, k, m->st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(loss, m->D.loss, sizeof(float), k, m->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->st);
    if (e != cudaSuccess) return mlp_map(e);
    return pic::mlp_take_error(m, m->st);
}

int pic_mlp_train(pic_mlp* m, int64_t n_data, const float* X_dev, const float* T_dev, int64_t batch, int64_t steps,
                  const pic_adam_t* opt, uint64_t seed, float* loss_hist) {
    if (!m || !opt || n_data < 1 || batch < 1 || batch > m->max_batch || batch > n_data || steps < 0 || !X_dev ||
        !T_dev)
        return PIC_ERR_INVALID_ARG;
    if (!(opt->lr > 0.f) || !(opt->beta1 >= 0.f && opt->beta1 < 1.f) || !(opt->beta2 >= 0.f && opt->beta2 < 1.f) ||
        !(opt->eps > 0.f))
        return PIC_ERR_INVALID_ARG;
    // a multiplier coprime with n_data near n_data times the golden ratio
    // (shifted by the seed): consecutive batch rows land far apart in the
    // data set, and the batches walk a fixed permutation of it
    long long mul = (long long)((double)n_data * 0.6180339887498949) + (long long)(seed % 1024ull);
    if (mul < 1) mul = 1;
    while (gcd_ll(mul, n_data) != 1) ++mul;
    cudaError_t e = cudaSuccess;
    for (long long s = 0; s < steps && e == cudaSuccess; ++s) {
        const long long first = (s * batch) % n_data;
        // the losses stay on the device until kLossHist of them, or the last, are in
        const long long at = s % pic::kLossHist;
        e = mlp_step(m, batch, X_dev, T_dev, first, mul, n_data, m->D.loss + at, 1, opt);
        if (e == cudaSuccess && loss_hist && (at == pic::kLossHist - 1 || s == steps - 1)) {
            e = cudaMemcpyAsync(loss_hist + (s - at), m->D.loss, sizeof(float) * (size_t)(at + 1),
                                cudaMemcpyDeviceToHost, m->st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(m->st);
        }
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->st);
    if (e != cudaSuccess) return mlp_map(e);
    return pic::mlp_take_error(m, m->st);
}

int pic_mlp_apply_gradient(pic_mlp* m, const float* grad, int ptr_kind, const pic_adam_t* opt) {
    if (!m || !grad || !opt || (ptr_kind != PIC_PTR_HOST && ptr_kind != PIC_PTR_DEVICE)) return PIC_ERR_INVALID_ARG;
    if (!(opt->lr > 0.f) || !(opt->beta1 >= 0.f && opt->beta1 < 1.f) || !(opt->beta2 >= 0.f && opt->beta2 < 1.f) ||
        !(opt->eps > 0.f))
        return PIC_ERR_INVALID_ARG;
    // the caller's gradient as the one partial the update kernel sums
    cudaError_t e = cudaMemcpyAsync(m->D.grad_part, grad, sizeof(float) * pic::kMParams,
                                    ptr_kind == PIC_PTR_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, m->st);
    if (e == cudaSuccess) {
        pic::AdamArgs A;
        std::memset(&A, 0, sizeof(A));
        m->t += 1;
        A.lr = opt->lr;
        A.beta1 = opt->beta1;
        A.beta2 = opt->beta2;
        A.eps = opt->eps;
        A.c1 = (float)(1.0 / (1.0 - std::pow((double)opt->beta1, (double)m->t)));
        A.c2 = (float)(1.0 / (1.0 - std::pow((double)opt->beta2, (double)m->t)));
        A.apply = 1;
        pic::k_mlp_update<<<pic::kUpdateBlocks, 128, 0, m->st>>>(m->D, 1, 0, m->D.loss, A);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->st);
    return mlp_map(e);
}

void pic_mlp_destroy(pic_mlp* m) {
    if (!m) return;
    cudaStreamSynchronize(m->st);
    mlp_free(m);
    delete m;
}

}  // extern "C"
