// mesh.cu -- standalone field-cycle kernels: CIC deposit, trapezoid prefix
// integral (decoupled look-back int64 scan) and gather (Sec. 2.3 of Frenod,
// Hirstoaga & Lutz; eq. VlasPoissAxSymBeam).
#include <algorithm>
#include <mutex>

#include "pic.h"
#include "pic_device.cuh"
#include "pic_internal.h"

namespace pic {

// ------------------------------------------------------------------ deposit

// Linear deposit of every particle as exact integers: floor(f W) units to
// the right node, W - floor(f W) to the left one.  Per-block histogram in
// shared memory when it fits, flushed with 64-bit integer atomics, so the
// result does not depend on the order of the additions.
template <int POW2>
__global__ void k_deposit(DevParams P, const double* __restrict__ R, long long n, int r_stride,
                          unsigned long long* __restrict__ Q, unsigned long long* __restrict__ n_out,
                          int use_smem) {
    extern __shared__ unsigned long long hist[];
    const int Np1 = P.n_cells + 1;
    if (use_smem) {
        for (int j = threadIdx.x; j < Np1; j += blockDim.x) hist[j] = 0ull;
        __syncthreads();
    }
    unsigned long long* H = use_smem ? hist : Q;
    unsigned int out = 0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        Cell c = mesh_locate<POW2>(P, R[i * r_stride]);
        if (c.j >= 0) {
            atomicAdd(&H[c.j], (unsigned long long)(P.W - c.qR));
            if (c.qR) atomicAdd(&H[c.j + 1], (unsigned long long)c.qR);
        } else {
            ++out;
        }
    }
    out = __reduce_add_sync(0xffffffffu, out);
    if ((threadIdx.x & 31) == 0 && out) atomicAdd(n_out, (unsigned long long)out);
    if (use_smem) {
        __syncthreads();
        for (int j = threadIdx.x; j < Np1; j += blockDim.x) {
            unsigned long long v = hist[j];
            if (v) atomicAdd(&Q[j], v);
        }
    }
}

// The same deposit with the binary32 quantisation of the FP32 form:
// x = (R - r_min)/h_r, j = floor(x), f = x - j and floor(f W) all in
// binary32 (W a power of two, so f W is exact).
__global__ void k_deposit32(DevParams P, const float* __restrict__ R, long long n, int r_stride,
                            unsigned long long* __restrict__ Q, unsigned long long* __restrict__ n_out, int use_smem) {
    extern __shared__ unsigned long long hist32[];
    const int Np1 = P.n_cells + 1;
    if (use_smem) {
        for (int j = threadIdx.x; j < Np1; j += blockDim.x) hist32[j] = 0ull;
        __syncthreads();
    }
    unsigned long long* H = use_smem ? hist32 : Q;
    unsigned int out = 0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const Cell32 c = locate32(P, R[i * r_stride]);
        if (c.j >= 0) {
            const unsigned long long qR = __float2ull_rz(c.a * P.Wf);
            atomicAdd(&H[c.j], (unsigned long long)P.W - qR);
            if (qR) atomicAdd(&H[c.j + 1], qR);
        } else {
            ++out;
        }
    }
    out = __reduce_add_sync(0xffffffffu, out);
    if ((threadIdx.x & 31) == 0 && out) atomicAdd(n_out, (unsigned long long)out);
    if (use_smem) {
        __syncthreads();
        for (int j = threadIdx.x; j < Np1; j += blockDim.x) {
            const unsigned long long v = hist32[j];
            if (v) atomicAdd(&Q[j], v);
        }
    }
}

// Split form of the deposit: W <= 2^32 and at most kSplitPositions positions
// per block.  Three 32-bit words per cell (count, low and high 16 bits of the
// right weights) stay exact for that many positions, and 32-bit shared
// reductions replace two 64-bit shared atomics per position; lane l deposits
// into copy l mod copies.  A block is a whole SM's threads, so that few blocks
// add to the mesh in global memory, and four positions per thread are in
// flight.  The 64-bit form (608 blocks of 256 threads, one position at a time)
// took 12.2 us for 10^6 positions on 256 cells, and stays for the rest.  With
// the field from one block (10 us in two launches before, and an allocation
// whose pool a synchronisation had emptied cost 200 us more) and four
// positions per thread in the gather (12.6 us before), a whole cycle of calls
// on 10^6 positions takes 24.6 us instead of 57.5.
constexpr int kSplitThreads = 1024;
constexpr long long kSplitPositions = 65536;
constexpr int kSplitAhead = 4;

__device__ __forceinline__ void split_add(unsigned int* h, int n_cells, int j, unsigned int q) {
    atomicAdd(&h[j], 1u);
    if (q & 0xffffu) atomicAdd(&h[n_cells + j], q & 0xffffu);
    if (q >> 16) atomicAdd(&h[2 * n_cells + j], q >> 16);
}

template <class Real, class Locate>
__device__ __forceinline__ void deposit_split(const DevParams& P, const Real* __restrict__ R, unsigned int n,
                                              int r_stride, unsigned long long* __restrict__ Q,
                                              unsigned long long* __restrict__ n_out, int copies, Locate locate) {
    extern __shared__ unsigned int split_hist[];  // copies x 3 x n_cells
    const int Nc = P.n_cells;
    for (int i = threadIdx.x; i < copies * 3 * Nc; i += blockDim.x) split_hist[i] = 0u;
    __syncthreads();
    unsigned int* h = split_hist + (threadIdx.x & (copies - 1)) * 3 * Nc;
    unsigned int out = 0;
    const unsigned int stride = gridDim.x * blockDim.x;
    for (unsigned long long i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (unsigned long long)kSplitAhead * stride) {
        Real r[kSplitAhead];
#pragma unroll
        for (int k = 0; k < kSplitAhead; ++k) {
            const unsigned long long m = i + (unsigned long long)k * stride;
            r[k] = m < n ? R[m * r_stride] : Real(0);
        }
#pragma unroll
        for (int k = 0; k < kSplitAhead; ++k) {
            if (i + (unsigned long long)k * stride >= n) break;
            int j;
            const unsigned int q = locate(r[k], j);
            if (j >= 0) split_add(h, Nc, j, q);
            else ++out;
        }
    }
    out = __reduce_add_sync(0xffffffffu, out);
    if ((threadIdx.x & 31) == 0 && out) atomicAdd(n_out, (unsigned long long)out);
    __syncthreads();
    // node charge Q_j = W C_j - S_j + S_{j-1}
    for (int j = threadIdx.x; j <= Nc; j += blockDim.x) {
        unsigned long long v = 0;
        for (int c = 0; c < copies; ++c) {
            const unsigned int* w = split_hist + c * 3 * Nc;
            if (j < Nc)
                v += (unsigned long long)w[j] * (unsigned long long)P.W -
                     (((unsigned long long)w[2 * Nc + j] << 16) + w[Nc + j]);
            if (j > 0) v += ((unsigned long long)w[2 * Nc + j - 1] << 16) + w[Nc + j - 1];
        }
        if (v) atomicAdd(&Q[j], v);
    }
}

template <int POW2>
__global__ void __launch_bounds__(kSplitThreads) k_deposit_split(DevParams P, const double* __restrict__ R,
                                                                 unsigned int n, int r_stride,
                                                                 unsigned long long* __restrict__ Q,
                                                                 unsigned long long* __restrict__ n_out, int copies) {
    deposit_split(P, R, n, r_stride, Q, n_out, copies, [&](double r, int& j) -> unsigned int {
        const Cell c = mesh_locate<POW2>(P, r);
        j = c.j;
        return (unsigned int)c.qR;
    });
}

__global__ void __launch_bounds__(kSplitThreads) k_deposit32_split(DevParams P, const float* __restrict__ R,
                                                                   unsigned int n, int r_stride,
                                                                   unsigned long long* __restrict__ Q,
                                                                   unsigned long long* __restrict__ n_out, int copies) {
    deposit_split(P, R, n, r_stride, Q, n_out, copies, [&](float r, int& j) -> unsigned int {
        const Cell32 c = locate32(P, r);
        j = c.j;
        return c.qR;
    });
}

__global__ void k_zero_charge(unsigned long long* __restrict__ Q, int n, unsigned long long* __restrict__ n_out) {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) Q[j] = 0ull;
    if (blockIdx.x == 0 && threadIdx.x == 0) *n_out = 0ull;
}

// ------------------------------------------------- field of a small mesh, one block
//
// S_j = G_j - G_c of every node (see below for G) by one block: warp w takes 32 R
// consecutive nodes, 32 at a time (coalesced), and scans them with shuffles.  No
// scratch, no status, no second launch up to kFieldFusedCells cells, where the
// block also evaluates the field.  Beyond, the ~13 FP64 operations per node (a
// division among them) would take one SM's pipe longer than a second launch:
// the block leaves S_j in E's own storage for k_field_in_place (and finishes the
// axis node, whose field is no S_j).  The line lies where R = 16 still fits the
// registers: 256 / 1024 / 4096 / 10000 cells take 4.6 / 8.2 / 12.4 / 14.4 us a call.
// The look-back form beyond it allocates scratch and waits for the host (34 us a
// call on these meshes, 200 us more after the pool was emptied).
constexpr int kFieldBlock = 1024;
constexpr int kFieldBlockCells = 16 * kFieldBlock - 2;
constexpr int kFieldFusedCells = 512;
static_assert(kFieldFusedCells < kFieldBlock, "one node per thread");

// E may be Q's own storage: neither is __restrict__, and E is accessed as its
// bits, in the type of Q.
__device__ __forceinline__ void field_node(const DevParams& P, const long long* Q, int j, long long S, long long* E,
                                           double* __restrict__ edges) {
    const int Nc = P.n_cells, c = P.c;
    double e;
    if (j == c) {
        e = P.parity_odd ? 0.0 : ((double)Q[c] * P.q_unit) * P.inv_hr;
    } else {
        const double r = P.r_min + (double)j * P.hr;
        e = ((double)S * P.q_half) * (1.0 / r);
        if (P.parity_odd && j < c) e = -e;  // odd reading: rE / |r|
    }
    E[j] = __double_as_longlong(e);
    // the off-mesh gather divides the edge rE by R; the odd reading's
    // lower edge carries the sign flip
    if (j == 0) edges[0] = P.parity_odd ? -((double)S * P.q_half) : (double)S * P.q_half;
    if (j == Nc) edges[1] = (double)S * P.q_half;
}

__device__ __forceinline__ long long warp_incl_scan(long long x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        long long y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    return x;
}

template <int R>
__global__ void __launch_bounds__(kFieldBlock) k_field_block(DevParams P, const long long* Q, long long* E,
                                                             double* __restrict__ edges, int fused) {
    __shared__ long long s_tot[kFieldBlock / 32], s_c;
    const int Nc = P.n_cells, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int j0 = w * 32 * R + lane;
    long long g[R], total = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int j = j0 + 32 * r;
        g[r] = j < Nc ? Q[j] + Q[j + 1] : 0ll;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const long long incl = warp_incl_scan(g[r]);
        g[r] = total + incl - g[r];
        total += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) s_tot[w] = total;
    __syncthreads();
    long long t = lane < w ? s_tot[lane] : 0ll;
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (j0 + 32 * r == P.c) s_c = t + g[r];
    __syncthreads();
    t -= s_c;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int j = j0 + 32 * r;
        if (j > Nc) break;
        if (R == 1 && fused) field_node(P, Q, j, t + g[r], E, edges);
        else if (j != P.c) E[j] = t + g[r];
    }
    if (!(R == 1 && fused) && threadIdx.x == 0) field_node(P, Q, P.c, 0ll, E, edges);
}

__global__ void k_field_in_place(DevParams P, const long long* Q, long long* E, double* __restrict__ edges) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j <= P.n_cells && j != P.c) field_node(P, Q, j, E[j], E, edges);
}

// ------------------------------------------------- decoupled look-back scan

__device__ __forceinline__ void st_release_s32(int* p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// G_j = sum_{m<j} (Q_m + Q_{m+1}), j = 0..n_cells, in one pass: each block
// scans a tile with warp shuffles, then its first thread looks back over
// the published aggregates/prefixes of earlier tiles (tiles are taken in
// launch order through an atomic counter, so every tile it waits on is
// already running).  Each wait has a time limit that sets the status word.
__global__ void __launch_bounds__(kScanThreads) k_scan_pairs(DevParams P, const long long* __restrict__ Q,
                                                             ScanScratch S) {
    __shared__ int s_tile;
    __shared__ long long s_warp[kScanThreads / 32];
    __shared__ long long s_excl;
    const int Nc = P.n_cells;
    if (threadIdx.x == 0) s_tile = (int)atomicAdd(S.tile_ctr, 1u);
    __syncthreads();
    const int tile = s_tile;
    const long long base = (long long)tile * kScanTile + (long long)threadIdx.x * kScanItems;
    long long v[kScanItems];
    long long sum = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        long long m = base + k;
        v[k] = (m < Nc) ? Q[m] + Q[m + 1] : 0;
        sum += v[k];
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long incl = warp_incl_scan(sum);
    if (lane == 31) s_warp[w] = incl;
    __syncthreads();
    if (w == 0) {
        long long y = (lane < kScanThreads / 32) ? s_warp[lane] : 0;
        y = warp_incl_scan(y);
        if (lane < kScanThreads / 32) s_warp[lane] = y;
    }
    __syncthreads();
    const long long total = s_warp[kScanThreads / 32 - 1];
    const long long in_block = incl - sum + (w > 0 ? s_warp[w - 1] : 0);
    if (threadIdx.x == 0) {
        long long excl = 0;
        if (tile == 0) {
            S.incl[0] = total;
            st_release_s32(&S.flag[0], 2);
        } else {
            S.agg[tile] = total;
            st_release_s32(&S.flag[tile], 1);
            int p = tile - 1;
            long long t0 = 0;
            unsigned spins = 0;
            while (p >= 0) {
                int f = ld_acquire_s32(&S.flag[p]);
                if (f == 2) {
                    excl += __ldcg(&S.incl[p]);
                    break;
                }
                if (f == 1) {
                    excl += __ldcg(&S.agg[p]);
                    --p;
                    continue;
                }
                if ((++spins & 63) == 0) {
                    long long now = global_ns();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > P.wait_ns) {
                        atomicCAS(S.status, 0, (int)DEV_TIMEOUT);
                        break;
                    }
                }
            }
            S.incl[tile] = excl + total;
            st_release_s32(&S.flag[tile], 2);
        }
        s_excl = excl;
    }
    __syncthreads();
    long long run = s_excl + in_block;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        long long m = base + k;
        if (m < Nc) {
            S.G[m] = run;
            if (m == Nc - 1) S.G[Nc] = run + v[k];
        }
        run += v[k];
    }
}

// S_j = G_j - G_c (the integral from r = 0), rE_j = S_j q_unit/2,
// E_j = rE_j * (1/r_j); at r = 0, E = rho(0) = Q_c q_unit / h_r.
__global__ void k_field_from_prefix(DevParams P, const long long* Q, const long long* __restrict__ G, long long* E,
                                    double* __restrict__ edges) {
    const long long Gc = G[P.c];
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j <= P.n_cells; j += gridDim.x * blockDim.x)
        field_node(P, Q, j, G[j] - Gc, E, edges);
}

// ------------------------------------------------------------------ gather

template <int POW2, int AHEAD>
__global__ void k_gather(DevParams P, const double* __restrict__ R, long long n,
                         const double* __restrict__ E, const double* __restrict__ edges,
                         double* __restrict__ out, int use_smem) {
    extern __shared__ double2 tab[];
    const int Nc = P.n_cells;
    if (use_smem) {
        for (int j = threadIdx.x; j < Nc; j += blockDim.x)
            tab[j] = make_double2(E[j], (E[j + 1] - E[j]) * P.invW);
        __syncthreads();
    }
    const double lo = edges[0], hi = edges[1];
    const long long stride = (long long)gridDim.x * blockDim.x;
    // AHEAD positions per thread in flight
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += AHEAD * stride) {
        double r[AHEAD];
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) r[k] = i + k * stride < n ? R[i + k * stride] : 0.0;
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) {
            if (i + k * stride >= n) break;
            const Cell c = mesh_locate<POW2>(P, r[k]);
            double e;
            if (use_smem) {
                e = mesh_gather(tab, lo, hi, c.j, c.a);
            } else if (c.j >= 0) {
                const double ej = E[c.j];
                e = fma(c.a, (E[c.j + 1] - ej) * P.invW, ej);
            } else {
                e = gather_outside(lo, hi, c.j, c.a);
            }
            out[i + k * stride] = e;
        }
    }
}

// ------------------------------------------------------------ (R, V) packing

__global__ void k_pack(const double* __restrict__ R, const double* __restrict__ V, double2* __restrict__ y,
                       long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = make_double2(R[i], V[i]);
}

__global__ void k_unpack(const double2* __restrict__ y, double* __restrict__ R, double* __restrict__ V,
                         long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double2 v = y[i];
        if (R) R[i] = v.x;
        if (V) V[i] = v.y;
    }
}

// y = y0 + N (y - y0) (eq. step2ClassicalETDAlgo), element by element.
__global__ void k_extrapolate_classic(double2* __restrict__ y, const double2* __restrict__ y0, long long n, double N) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double2 a = y0[i], b = y[i];
        y[i] = make_double2(a.x + N * (b.x - a.x), a.y + N * (b.y - a.y));
    }
}

// ------------------------------------------------------------ host launchers

static int grid_for(long long n, int sm_count) {
    long long want = (n + 255) / 256;
    long long cap = (long long)sm_count * 8;
    return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

cudaError_t launch_extrapolate_classic(double2* y, const double2* y0, long long n, double N, int sm_count,
                                       cudaStream_t st, long long* launches) {
    if (n == 0) return cudaSuccess;
    k_extrapolate_classic<<<grid_for(n, sm_count), 256, 0, st>>>(y, y0, n, N);
    if (launches) ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_pack(const double* R, const double* V, double2* y, long long n, int sm_count, cudaStream_t st,
                        long long* launches) {
    if (n == 0) return cudaSuccess;
    k_pack<<<grid_for(n, sm_count), 256, 0, st>>>(R, V, y, n);
    if (launches) ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_unpack(const double2* y, double* R, double* V, long long n, int sm_count, cudaStream_t st,
                          long long* launches) {
    if (n == 0) return cudaSuccess;
    k_unpack<<<grid_for(n, sm_count), 256, 0, st>>>(y, R, V, n);
    if (launches) ++*launches;
    return cudaGetLastError();
}

// Shared memory that a block's histograms or field table may take.  A kernel that
// needs more than the 48 KB it has without asking is given all of it: the limit is
// the kernel's, and a thread that set its own mesh's size could lower it between
// another thread's setting and launch.
constexpr size_t kMeshSmem = 96 * 1024;
static cudaError_t open_mesh_smem(const void* fn, size_t smem) {
    return smem > 48 * 1024 ? cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMeshSmem)
                            : cudaSuccess;
}

// Zeroed charge and out-of-mesh count, then the split form where it serves
// (its histograms of 12 bytes per cell and copy within 48 KB, or 96 KB with one
// copy), else the 64-bit form.
template <class Real, class Split, class Wide>
static cudaError_t deposit_with(Split split_fn, Wide wide_fn, const DevParams& P, const Real* R, long long n, int r_stride,
                                long long* Q, long long* n_out, cudaStream_t st, int sm_count, long long* launches) {
    const int Np1 = P.n_cells + 1;
    k_zero_charge<<<(Np1 + 255) / 256, 256, 0, st>>>((unsigned long long*)Q, Np1, (unsigned long long*)n_out);
    if (launches) ++*launches;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || n == 0) return e;
    const size_t per_copy = sizeof(unsigned int) * 3 * (size_t)P.n_cells;
    if (P.W <= (1ll << 32) && per_copy <= kMeshSmem && n < (1ll << 31)) {
        const int copies = 4 * per_copy <= 48 * 1024 ? 4 : (2 * per_copy <= 48 * 1024 ? 2 : 1);
        const size_t smem = copies * per_copy;
        if ((e = open_mesh_smem((const void*)split_fn, smem)) != cudaSuccess) return e;
        // one block per SM, or as many full waves of them as keep every block
        // within its positions (whole rounds of kSplitThreads positions each).  The
        // least number of blocks instead left 2 of 306 to a wave of their own: 2 10^7
        // positions on 1000 cells took 238 us, now 166 (64-bit form 167); on 256
        // cells 117, now 84 (64-bit form 126).
        const long long rounds = (n + kSplitThreads - 1) / kSplitThreads, most = kSplitPositions / kSplitThreads;
        const long long waves = (rounds + most * sm_count - 1) / (most * sm_count);
        const long long grid = rounds < sm_count ? rounds : waves * sm_count;
        split_fn<<<(int)grid, kSplitThreads, smem, st>>>(P, R, (unsigned int)n, r_stride, (unsigned long long*)Q,
                                                         (unsigned long long*)n_out, copies);
    } else {
        const size_t smem = sizeof(unsigned long long) * (size_t)Np1;
        const int use_smem = smem <= kMeshSmem;
        if (use_smem && (e = open_mesh_smem((const void*)wide_fn, smem)) != cudaSuccess) return e;
        const long long want = (n + 255) / 256;
        const int grid = (int)(want < (long long)sm_count * 4 ? want : (long long)sm_count * 4);
        wide_fn<<<grid, 256, use_smem ? smem : 0, st>>>(P, R, n, r_stride, (unsigned long long*)Q,
                                                        (unsigned long long*)n_out, use_smem);
    }
    if (launches) ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_deposit(const DevParams& P, const double* R, long long n, int r_stride, long long* Q,
                           long long* n_out, cudaStream_t st, int sm_count, long long* launches) {
    return P.xs_fma ? deposit_with(k_deposit_split<1>, k_deposit<1>, P, R, n, r_stride, Q, n_out, st, sm_count, launches)
                    : deposit_with(k_deposit_split<0>, k_deposit<0>, P, R, n, r_stride, Q, n_out, st, sm_count, launches);
}

cudaError_t launch_deposit32(const DevParams& P, const float* R, long long n, int r_stride, long long* Q,
                             long long* n_out, cudaStream_t st, int sm_count, long long* launches) {
    return deposit_with(k_deposit32_split, k_deposit32, P, R, n, r_stride, Q, n_out, st, sm_count, launches);
}

size_t scan_scratch_bytes(int n_cells) {
    const int tiles = (n_cells + kScanTile - 1) / kScanTile;
    return scan_scratch_layout(n_cells, tiles, nullptr, nullptr);
}

size_t scan_scratch_layout(int n_cells, int tiles, void* base, ScanScratch* S) {
    // agg, incl (tiles int64 each), G (n_cells+1 int64), flag (tiles int32),
    // tile counter and status (int32 each); every piece 256-byte aligned.
    auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
    size_t off_agg = 0;
    size_t off_incl = up(off_agg + sizeof(long long) * tiles);
    size_t off_G = up(off_incl + sizeof(long long) * tiles);
    size_t off_flag = up(off_G + sizeof(long long) * (size_t)(n_cells + 1));
    size_t off_ctr = up(off_flag + sizeof(int) * tiles);
    size_t off_status = up(off_ctr + sizeof(unsigned int));
    size_t total = up(off_status + sizeof(int));
    if (S && base) {
        char* b = (char*)base;
        S->agg = (long long*)(b + off_agg);
        S->incl = (long long*)(b + off_incl);
        S->G = (long long*)(b + off_G);
        S->flag = (int*)(b + off_flag);
        S->tile_ctr = (unsigned int*)(b + off_ctr);
        S->status = (int*)(b + off_status);
        S->zero_from = off_flag;  // flags, counter and status must start at zero
        S->zero_bytes = total - off_flag;
    }
    return total;
}

bool poisson_in_block(int n_cells) { return n_cells <= kFieldBlockCells; }

cudaError_t launch_poisson(const DevParams& P, const long long* Q, double* E, double* edges,
                           const ScanScratch& S, cudaStream_t st, long long* launches) {
    long long* const Eb = (long long*)E;  // as bits (field_node)
    if (poisson_in_block(P.n_cells)) {
        const int fused = P.n_cells <= kFieldFusedCells;
        if (P.n_cells < kFieldBlock) k_field_block<1><<<1, kFieldBlock, 0, st>>>(P, Q, Eb, edges, fused);
        else if (P.n_cells < 4 * kFieldBlock) k_field_block<4><<<1, kFieldBlock, 0, st>>>(P, Q, Eb, edges, fused);
        else k_field_block<16><<<1, kFieldBlock, 0, st>>>(P, Q, Eb, edges, fused);
        if (!fused) k_field_in_place<<<(P.n_cells + 256) / 256, 256, 0, st>>>(P, Q, Eb, edges);
        if (launches) *launches += fused ? 1 : 2;
        return cudaGetLastError();
    }
    const int tiles = (P.n_cells + kScanTile - 1) / kScanTile;
    cudaError_t e = cudaMemsetAsync((char*)S.flag, 0, S.zero_bytes, st);
    if (e != cudaSuccess) return e;
    k_scan_pairs<<<tiles, kScanThreads, 0, st>>>(P, Q, S);
    int fgrid = (P.n_cells + 1 + 255) / 256;
    k_field_from_prefix<<<fgrid, 256, 0, st>>>(P, Q, S.G, Eb, edges);
    if (launches) *launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_gather(const DevParams& P, const double* R, long long n, const double* E,
                          const double* edges, double* out, cudaStream_t st, int sm_count,
                          long long* launches) {
    if (n == 0) return cudaSuccess;
    size_t smem = sizeof(double2) * (size_t)P.n_cells;
    int use_smem = smem <= kMeshSmem;
    // Without a table the loads of E go to L2, and one position at a time in four
    // blocks per SM is as fast or faster up to 36 positions per thread (5.6 10^6).  One /
    // four in flight on 65536 cells: 10^6 positions 10.3 / 11.7 us, 2 10^6 16.5 / 18.2,
    // 4 10^6 28.8 / 29.1, 6 10^6 45.2 / 43.2, 8 10^6 66.4 / 57.8, 2 10^7 157 / 145.
    const int one = !use_smem && n <= 36ll * 4 * 256 * sm_count;
    auto fn = one ? (P.xs_fma ? k_gather<1, 1> : k_gather<0, 1>) : (P.xs_fma ? k_gather<1, 4> : k_gather<0, 4>);
    if (use_smem) {
        const cudaError_t e = open_mesh_smem((const void*)fn, smem);
        if (e != cudaSuccess) return e;
    }
    long long want = (n + 255) / 256;
    // one position per thread while the GPU has room, then four in flight.  Each block
    // builds its table (two FP64 operations per cell, about a quarter of four
    // positions'), so the blocks per SM follow the positions per cell.
    // (10^6 positions on 4096 cells: 977 blocks 30.8 us, 608 blocks 26.6, 304
    // 16.5; 10^5 on 256 cells: 98 blocks 6.2, 391 blocks 5.1.)  Without a table eight
    // blocks pay for the largest sets only (four / eight with four in flight: 6 10^6 43.2 /
    // 48.4 us, 8 10^6 57.8 / 62.2).
    const long long per_sm = use_smem ? std::min(8ll, 2 + n / (4ll * sm_count * P.n_cells)) : (n < (1ll << 23) ? 4 : 8);
    const int grid = (int)std::min(want, per_sm * sm_count);
    fn<<<grid, 256, use_smem ? smem : 0, st>>>(P, R, n, E, edges, out, use_smem);
    if (launches) ++*launches;
    return cudaGetLastError();
}

}  // namespace pic

// ----------------------------------------------- scan without allocation

namespace pic {

// Fixed device scratch for pic_poisson_noalloc: the look-back tile states,
// the prefix G and the status word of one scan of at most
// kNoAllocMaxCells cells.  Every GPU that loads the library holds it until
// the process exits.
constexpr int kNoAllocMaxCells = 16384;
constexpr size_t kNoAllocScratchBytes = 136 * 1024;
static __device__ __align__(256) unsigned char g_poisson_scratch[kNoAllocScratchBytes];

}  // namespace pic

extern "C" int pic_poisson_noalloc(const pic_params* p, int64_t n_particles, const int64_t* Q_dev, double* E_dev,
                                   double* rE_edges_dev, void* stream) {
    // Host code cannot use g_poisson_scratch's name as a device address: the
    // address is looked up once per device (with that device current) and
    // cached.  This set-up happens in the first call on each device.
    static std::mutex mu;
    static void* scratch_addr[256] = {};
    if (!p) return PIC_ERR_INVALID_ARG;
    // a mesh too small for the layout arithmetic below is a bad argument
    // (the full parameter check runs in the shared body)
    if (p->n_cells < 2) return PIC_ERR_INVALID_ARG;
    if (p->n_cells > pic::kNoAllocMaxCells) return PIC_ERR_TOO_LARGE;
    if (n_particles <= 0 || !Q_dev || !E_dev || !rE_edges_dev) return PIC_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return PIC_ERR_CUDA;
    void* base = nullptr;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!scratch_addr[dev]) {
            void* a = nullptr;
            if (cudaGetSymbolAddress(&a, pic::g_poisson_scratch) != cudaSuccess || !a) return PIC_ERR_CUDA;
            scratch_addr[dev] = a;
        }
        base = scratch_addr[dev];
    }
    const int tiles = (p->n_cells + pic::kScanTile - 1) / pic::kScanTile;
    if (pic::scan_scratch_layout(p->n_cells, tiles, nullptr, nullptr) > pic::kNoAllocScratchBytes) return PIC_ERR_TOO_LARGE;
    pic::ScanScratch S;
    pic::scan_scratch_layout(p->n_cells, tiles, base, &S);
    const int rc = pic::poisson_with_scratch(p, n_particles, Q_dev, E_dev, rE_edges_dev, &S, stream);
    // this entry point returns with the field solved for every mesh it takes
    if (rc == PIC_OK && pic::poisson_in_block(p->n_cells) && cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess)
        return PIC_ERR_CUDA;
    return rc;
}
