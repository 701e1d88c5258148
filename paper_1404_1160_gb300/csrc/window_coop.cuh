// window_coop.cuh -- the cooperative window kernel of the Poisson field
// (k_window_coop) and its device helpers, included by window_coop.cu, which
// is compiled once per histogram form and fine solver (the instantiations
// compile in parallel), and by window.cu for the launch sizes.
//
// The fine window of Algorithm ETDFSSModAlgo (Frenod, Hirstoaga
// & Lutz, Sec. 3): fine solver from y^n with period detection (Remark
// CompOfThePeriodsRem), quadratic landing at o and o+T (Remark
// QuadraticInterpolationRem) and the N-turn extrapolation (eq. MainFormula1).
//
// Self-consistent Poisson field: one cooperative persistent launch per macro
// step.  Each fine stage needs the field of every particle's stage position
// (Sec. 3: the window advances every particle, not only those still
// looking for their period, because the self-consistent field needs them
// all).  Because E enters only dV/dt, the
// R-component of stage s depends on fields of stages <= s-2, so stages pair
// up: RK4 deposits stages (1,2) then (3,4); Lawson RK4 deposits (1,3) then
// (2,4).  One fine step is therefore two field cycles:
//   sweep: gather previous pair, advance, deposit the next pair into a
//          shared-memory int64 histogram per block;
//   add the histograms to the cycle's global charge words and wait until
//   every block has (window_common.cuh);
//   every block scans the mesh charge (block-wide int64 scan) into its own
//   shared-memory field table.
#pragma once

#include "pic_internal.h"
#include "window_common.cuh"

namespace pic {

constexpr int kWinMaxThreads = 1024;
constexpr int kHistCopiesMax = 2;

// ---------------------------------------------------------------- helpers

// Shared-memory histogram of one field.  HIST = 0: three 32-bit counters
// per cell (particles C_j, low and high 16 bits of the right weights S_j),
// exact while a block deposits at most 65536 positions per field per cycle;
// the node charge is Q_j = W C_j - S_j + S_{j-1}.  HIST = 2: four counters
// (C_j and the 11/11/10-bit parts of S_j), exact up to 2^21 positions per
// block, field and cycle, for the larger particle counts.  HIST = 1: one
// 64-bit counter per node (W > 2^32, or beyond 2^21 positions).
template <int HIST>
struct Hist {
    static constexpr int kWordsPerNode = HIST == 0 ? 3 : (HIST == 2 ? 4 : 2);  // 32-bit words per node
};
// 32-bit words per node that the shared-memory layout reserves
__host__ __device__ constexpr int hist_slot_words(int hist) { return hist == 2 ? 4 : 3; }

// histogram copies that the layout reserves: the staged field build uses the
// region as its int64 scan input, which takes two copies' words
__host__ __device__ constexpr int hist_copies_reserved(int n_cells, int copies, int block) {
    return copies < 2 && !field_in_regs(n_cells, block) ? 2 : copies;
}

template <int HIST>
__device__ __forceinline__ void deposit_cell(unsigned int* h, int Np1, const Cell& c, long long W) {
    if (c.j < 0) return;
    if (HIST == 0) {
        // every lane adds its own position (plain shared atomics are faster
        // on this GPU than merging the lanes of a warp first)
        const unsigned int lo = (unsigned int)(c.qR & 0xffff), hi = (unsigned int)(c.qR >> 16);
        atomicAdd(&h[c.j], 1u);
        if (lo) atomicAdd(&h[Np1 + c.j], lo);
        if (hi) atomicAdd(&h[2 * Np1 + c.j], hi);
    } else if (HIST == 2) {
        const unsigned int q = (unsigned int)c.qR;
        const unsigned int a = q & 0x7ffu, b = (q >> 11) & 0x7ffu, d = q >> 22;
        atomicAdd(&h[c.j], 1u);
        if (a) atomicAdd(&h[Np1 + c.j], a);
        if (b) atomicAdd(&h[2 * Np1 + c.j], b);
        if (d) atomicAdd(&h[3 * Np1 + c.j], d);
    } else {
        unsigned long long* h64 = (unsigned long long*)h;
        atomicAdd(&h64[c.j], (unsigned long long)(W - c.qR));
        if (c.qR) atomicAdd(&h64[c.j + 1], (unsigned long long)c.qR);
    }
}

// Node charge of one field from the block histogram, summed over its
// `copies` copies `stride` words apart (lane l deposits into copy
// l % copies, so a cell shared by the lanes of a warp is updated on
// several addresses instead of one).
template <int HIST>
__device__ __forceinline__ unsigned long long hist_node(const unsigned int* h, int Np1, int j, long long W, int stride,
                                                        int copies) {
    if (HIST == 0) {
        unsigned long long C = 0, Sj = 0, Sm = 0;
        for (int c = 0; c < copies; ++c) {
            const unsigned int* hc = h + c * stride;
            if (j < Np1 - 1) {
                C += hc[j];
                Sj += ((unsigned long long)hc[2 * Np1 + j] << 16) + (unsigned long long)hc[Np1 + j];
            }
            if (j >= 1) Sm += ((unsigned long long)hc[2 * Np1 + j - 1] << 16) + (unsigned long long)hc[Np1 + j - 1];
        }
        return C * (unsigned long long)W - Sj + Sm;
    } else if (HIST == 2) {
        auto S = [&](const unsigned int* hc, int m) -> unsigned long long {
            return (unsigned long long)hc[Np1 + m] + ((unsigned long long)hc[2 * Np1 + m] << 11) +
                   ((unsigned long long)hc[3 * Np1 + m] << 22);
        };
        unsigned long long C = 0, Sj = 0, Sm = 0;
        for (int c = 0; c < copies; ++c) {
            const unsigned int* hc = h + c * stride;
            if (j < Np1 - 1) {
                C += hc[j];
                Sj += S(hc, j);
            }
            if (j >= 1) Sm += S(hc, j - 1);
        }
        return C * (unsigned long long)W - Sj + Sm;
    } else {
        return ((const unsigned long long*)h)[j];
    }
}

// Field tables of one cycle (two fields) from the cycle's global charge:
// trapezoid integral from r = 0 (S_j = g_j - g_c), E_j = S_j q_unit/2 * (1/r_j),
// E_c = Q_c q_unit / h_r, then (E_j, (E_{j+1}-E_j)/W) per cell.
// `control`: the cycle carries the not-done count; s_stop = (count == 0).
// One call ends a sweep: the block's histograms into the cycle's words, the
// table from the words of all blocks, and the histograms and the sweep's
// counters cleared for the next sweep.  false: a wait ran out of time.
struct NodeField {
    double E, rE;
};
static __device__ __forceinline__ NodeField shfl_next(const NodeField& v) {
    return {__shfl_down_sync(0xffffffffu, v.E, 1), v.rE};  // only E is used of the next lane's node
}

template <int HIST>
static __device__ __forceinline__ bool field_cycle(int cyc, bool control) {
    __syncthreads();
    const int Nc = s_cyc.n_cells, Np1 = Nc + 1, c = s_cyc.c, copies = s_cyc.copies;
    const int words = Hist<HIST>::kWordsPerNode * Np1;
    unsigned int* hist = (unsigned int*)(smem_raw + s_cyc.hist);
    double2* tab = (double2*)(smem_raw + s_cyc.tabA);
    const double* node_k = (const double*)(smem_raw + s_cyc.node_c);
    unsigned long long* prev;
    const unsigned long long* Q = cycle_exchange(cyc, control, &prev, [&](int f, int j) {
        return hist_node<HIST>(hist + f * words, Np1, j, s_cyc.W, 2 * words, copies);
    });
    if (!Q) return false;
    auto clear = [&]() {
        for (int i = threadIdx.x; i < copies * 2 * words; i += blockDim.x) hist[i] = 0u;
        if (threadIdx.x == 0) {
            s_cnt = 0;
            s_next = 0;
        }
    };
    // E_j = (S_j q_unit/2) (1/r_j), E_c = (Q_c q_unit) (1/h_r); node_k[c] is 1/h_r,
    // and with the odd reading (rE / |r|) 0 there and -1/r_j left of it.  One
    // code path for all nodes.
    auto field_at = [&](int j, long long S, long long qj) -> NodeField {
        NodeField v;
        v.rE = i64_to_double(j == c ? qj : S) * (j == c ? s_cyc.q_unit : s_cyc.q_half);
        v.E = v.rE * node_k[j];
        return v;
    };
    auto slope = [&](double d) -> double {
        // d / W: exponent shift when the result stays normal (exact), else multiply
        const int ex = (int)((__double_as_longlong(d) >> 52) & 0x7ff);
        return (ex > s_cyc.log2W + 1 && ex < 0x7ff) ? scale_pow2(d, -s_cyc.log2W) : d * s_cyc.invW;
    };
    auto edge = [&](int f, int j, double rE) {
        // the off-mesh gather divides the edge rE by R: the odd reading
        // (rE / |R|) carries the sign flip in the lower edge value
        if (j == 0) s_cyc.edges[2 * f] = s_cyc.parity_odd ? -rE : rE;
        if (j == Nc) s_cyc.edges[2 * f + 1] = rE;
    };
    if (field_in_regs(Nc, blockDim.x)) {
        auto emit = [&](int f, int j, const NodeField& v, const NodeField& next) {
            tab[f * Np1 + j] = make_double2(v.E, j < Nc ? slope(next.E - v.E) : 0.0);
            edge(f, j, v.rE);
        };
        if (!field_build_regs(Q, prev, control, field_at, emit, clear)) return false;
        __syncthreads();
        return true;
    }
    // staged build (meshes too large for the register form); the grid
    // barrier has put every thread past its flush, so q may take the histograms
    long long* q = (long long*)hist;
    long long* g = (long long*)(smem_raw + s_cyc.g);
    stage_charge(Q, q, control);
    __syncthreads();
    block_exscan_pairs2(q, g, Nc, s_tot);
    for (int idx = threadIdx.x; idx < 2 * Np1; idx += blockDim.x) {
        const int f = idx >= Np1, j = idx - f * Np1;
        const long long S = g[idx] - g[f * Np1 + c];
        const NodeField v = field_at(j, S, q[f * Np1 + c]);
        tab[idx].x = v.E;
        edge(f, j, v.rE);
    }
    __syncthreads();
    clear();
    for (int idx = threadIdx.x; idx < 2 * Np1; idx += blockDim.x) {
        const int f = idx >= Np1, j = idx - f * Np1;
        tab[idx].y = j < Nc ? slope(tab[idx + 1].x - tab[idx].x) : 0.0;
    }
    __syncthreads();
    return true;
}

// The third extremum (roots and resolution) or the window cap at sample k.
static __device__ __noinline__ int2 track_resolved(const DevParams& P, const WinBufs& B, unsigned int i, int k,
                                                   double Vold, double Vnew, bool detect_only, int2 tr) {
    Track s;
    s.flags = tr.x;
    if ((tr.x & F_NEXT) == 3) {
        const double v2 = detect_only ? B.traj[(size_t)(tr.y + 2) * P.n + i].y : B.o[i];
        const double t1 = (double)tr.y + quad_root01(B.t1[i], B.T[i], v2);
        s.T = ((double)(k - 2) + quad_root01(B.vp[i], Vold, Vnew)) - t1;
    } else {
        s.flags |= F_FB;
        s.T = P.Tfb;
    }
    if (detect_only) {
        s.flags |= F_RES;
        s.need = 0;
    } else {
        track_resolve(s, P, s.T);
        B.o[i] = s.o;
        B.N[i] = s.N;
    }
    B.T[i] = s.T;
    return make_int2(s.flags, s.need);
}

// Period tracking of one particle at sample k (k >= 1), V_{k-1} = Vold,
// V_k = Vnew.  A sign change between samples k-1 and k is marked pending
// (V_{k-1} kept in vp) and counted as an extremum at sample k+1, when its
// stencil V_{k-1}, V_k, V_{k+1} is complete: the same crossings, stencils and
// order as testing samples k-2, k-1 at sample k.  Only the third extremum
// evaluates roots: the first one keeps its stencil (in t1, T and o, which
// the resolution overwrites, and its sample in the word that later holds
// `need`), the second one needs no time.  A root and a resolution are chains
// of FP64 divisions, and one particle's holds up its block's sweep and with
// it every block's cycle; this way no cycle before the first full turn has
// one (with the table's single code path: FP64 10^6 particles 9.47 -> 9.03
// ms, the modified scheme on 150001 8.07 -> 7.40 ms).  tr = (flags, need) is loaded by the caller and updated here.
// Returns true when the particle is done.
__device__ __forceinline__ bool track_update(const DevParams& P, const WinBufs& B, unsigned int i, int k,
                                             double Vold, double Vnew, bool detect_only, int2& tr) {
    if (!(tr.x & F_RES)) {
        const bool pend = tr.x & F_PEND, change = positive(Vold) != positive(Vnew);
        if (pend || change || k == P.Kmax) {
            if (pend) {
                tr.x += 1 - F_PEND;
                if ((tr.x & F_NEXT) == 1) {
                    B.t1[i] = B.vp[i];
                    B.T[i] = Vold;
                    if (!detect_only) B.o[i] = Vnew;  // step 1 alone leaves o as it was; its rows hold the sample
                    tr.y = k - 2;
                }
            }
            if ((tr.x & F_NEXT) == 3 || k == P.Kmax) {
                tr = track_resolved(P, B, i, k, Vold, Vnew, detect_only, tr);
            } else if (change) {
                tr.x |= F_PEND;
                B.vp[i] = Vold;
            }
            B.tr[i] = tr;
        }
    }
    if (!(tr.x & F_RES)) return false;
    return detect_only || k >= tr.y;
}

// Trajectory band of an ETD window.  The landing reads rows floor(o) .. +2
// and floor(o + T) .. +2; with the previous step's period as the forecast
// of T, a window stores row 0 (y^n) and the rows within band_m of the two
// forecast stencils only.  The first rows of the two bands sit in bits
// 8..19 and 20..31 of the tracking word (the flags use bits 0..4).
__device__ __forceinline__ int band_bits(const DevParams& P, double Tprev) {
    const double T = (Tprev > 0.0 && isfinite(Tprev)) ? Tprev : P.Tfb;
    const double o = fmod(P.D, T);
    const int N = (int)rint((P.D - o) / T);
    int a = (int)floor(o) - P.band_m, b = N > 0 ? (int)floor(o + T) - P.band_m : a;
    a = min(max(a, 0), 4095);
    b = min(max(b, 0), 4095);
    return (int)(((unsigned int)a << 8) | ((unsigned int)b << 20));
}
__device__ __forceinline__ bool band_holds(int x, int k, int band_m) {
    const unsigned int ux = (unsigned int)x, L = 3u + 2u * (unsigned int)band_m;
    return k == 0 || (unsigned int)(k - (int)((ux >> 8) & 0xFFFu)) < L || (unsigned int)(k - (int)(ux >> 20)) < L;
}

// ------------------------------------------------ cooperative Poisson window

// One chunk (32 particles) of window state in shared memory; lane l owns
// entry l of every array, so no warp synchronisation is needed.  cx: Lawson
// carries (Phi_h y)_R, RK4 both stage positions.
template <int SOLVER>
struct StageCx {
    double2 cx[32];
};
template <>
struct StageCx<1> {
    double cx[32];
};
template <int SOLVER>
struct Stage : StageCx<SOLVER> {
    double2 y[32];
    double2 ce[32];
    double2 ca[32];
    int2 tr[32];
    short2 cj[32];
};
// How a window keeps its chunks: in global memory, loaded directly (0) or
// through a double buffer per warp (1: the next chunk is in flight while the
// current one is worked on), or in shared memory for the whole window (2).
// A resident chunk saves the L2 round trip at the start of every sweep,
// which a beam with one or two chunks per warp cannot hide.  Measured on
// GB300 together with one block per SM instead of n/1024 blocks: two RK4 steps
// of 20000 particles 9.17 -> 5.79 ms, the modified scheme on 150001 8.64 ->
// 8.07 ms; 10^6 particles do not fit and stay staged (9.5 ms).
enum WindowStage { STAGE_NONE = 0, STAGE_NEXT = 1, STAGE_RESIDENT = 2 };
// Chunk buffers a block holds; `chunks`: the chunks of one block.
__host__ __device__ constexpr size_t stage_buffers(int stage, int block, unsigned int chunks) {
    return stage == STAGE_RESIDENT ? chunks : (stage == STAGE_NEXT ? 2 * (size_t)(block >> 5) : 0);
}

// The state a sweep reads for one particle.
struct ChunkIn {
    double2 y, ce, ca, cx;
    int2 tr;
    short2 cj;
};

template <int SOLVER>
__device__ __forceinline__ void prefetch_chunk(const WinBufs& B, unsigned int i, bool sweepA, bool fine_only, bool k0,
                                               Stage<SOLVER>* s, int lane) {
    cp_async16(&s->y[lane], &B.y[i]);
    if (sweepA && !fine_only) cp_async8(&s->tr[lane], &B.tr[i]);
    if (sweepA && k0) return;
    if (sweepA) cp_async16(&s->ce[lane], &B.ce[i]);
    cp_async16(&s->ca[lane], &B.ca[i]);
    if constexpr (SOLVER == 1) cp_async8(&s->cx[lane], &B.cxr[i]);
    else cp_async16(&s->cx[lane], &B.cx[i]);
    cp_async4(&s->cj[lane], &B.cj[i]);
}

template <int SOLVER>
__device__ __forceinline__ ChunkIn load_chunk(const WinBufs& B, unsigned int i, bool sweepA, bool fine_only, bool k0) {
    ChunkIn c;
    c.y = B.y[i];
    c.tr = (sweepA && !fine_only) ? B.tr[i] : make_int2(0, 0);
    c.ce = make_double2(0.0, 0.0);
    c.ca = make_double2(0.0, 0.0);
    c.cx = make_double2(0.0, 0.0);
    c.cj = make_short2(-3, -3);
    if (sweepA && k0) return c;
    if (sweepA) c.ce = B.ce[i];
    c.ca = B.ca[i];
    if (SOLVER == 1) c.cx.x = B.cxr[i];
    else c.cx = B.cx[i];
    c.cj = B.cj[i];
    return c;
}

template <int SOLVER>
__device__ __forceinline__ ChunkIn read_stage(const Stage<SOLVER>* s, int lane) {
    ChunkIn c;
    c.y = s->y[lane];
    c.ce = s->ce[lane];
    c.ca = s->ca[lane];
    if constexpr (SOLVER == 1) c.cx = make_double2(s->cx[lane], 0.0);
    else c.cx = s->cx[lane];
    c.tr = s->tr[lane];
    c.cj = s->cj[lane];
    return c;
}

template <int SOLVER, int HIST, int POW2, int STAGE>
__global__ void __launch_bounds__(kWinMaxThreads) k_window_coop(DevParams P, WinBufs B, int mode, int T_known,
                                                                long long n_fine, const double* __restrict__ Tin) {
    const int Nc = P.n_cells, Np1 = Nc + 1;
    const int words = Hist<HIST>::kWordsPerNode * Np1;   // 32-bit words per field histogram
    const int copies = P.hist_copies;
    const unsigned int n = (unsigned int)P.n;             // below 2^31
    const unsigned int n_chunks = (n + 31) / 32;
    Stage<SOLVER>* stage = (Stage<SOLVER>*)smem_raw;
    double2* tab = (double2*)(stage + stage_buffers(STAGE, blockDim.x, (n_chunks + gridDim.x - 1) / gridDim.x));  // 2 Np1
    unsigned int* hist = (unsigned int*)(tab + 2 * Np1);  // copies x 2 fields x words (staged build: also the scan input)
    long long* g = (long long*)(hist + hist_copies_reserved(Nc, copies, blockDim.x) * 2 * hist_slot_words(HIST) * Np1);  // 2 Np1
    double* node_k = (double*)(g + cycle_words(Nc, blockDim.x, P.q_cb > 0));  // Np1
    // the region of g holds the last complete charge words of the two slots
    // instead where the field is built in registers
    unsigned long long* prev = (unsigned long long*)g;  // 2 x (2 Np1 + 1)
    if (P.q_cb)
        for (int i = threadIdx.x; i < 2 * (2 * Np1 + 1); i += blockDim.x) prev[i] = 0ull;
    for (int i = threadIdx.x; i < copies * 2 * words; i += blockDim.x) hist[i] = 0u;
    auto off = [&](const void* p) { return (int)((const unsigned char*)p - smem_raw); };
    cycle_setup(P, B.Qring, B.bar, B.status, gridDim.x, blockIdx.x, off(hist), off(tab), 0, off(g), off(node_k));
    for (int j = threadIdx.x; j < Np1; j += blockDim.x)
        node_k[j] = j == P.c ? (P.parity_odd ? 0.0 : P.inv_hr)
                             : ((P.parity_odd && j < P.c) ? -1.0 : 1.0) / (P.r_min + (double)j * P.hr);

    const bool detect_only = mode == MODE_PERIODS, fine_only = mode == MODE_FINE;
    // Work unit: a chunk of 32 consecutive storage slots (phase-space
    // neighbours after the sort).  Block b owns the chunks c = b (mod grid),
    // so every block sees all phases (the sign changes of V spread evenly
    // over blocks and fine steps) and a slot always stays on one SM; inside
    // the block, warps take the block's chunks dynamically from a shared
    // counter, so they finish a sweep together.
    const int lane = threadIdx.x & 31;
    const unsigned int my_chunks = blockIdx.x < n_chunks ? (n_chunks - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    // lane l deposits into copy l mod copies (the lanes of a warp hold
    // phase-space neighbours, which mostly share a cell)
    unsigned int* const my_hist = hist + ((threadIdx.x & 31) % copies) * 2 * words;
    const unsigned int warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    Stage<SOLVER>* const my_stage = stage + 2 * warp;  // STAGE_NEXT
    // Chunk m of this block starts at slot 32 (blockIdx.x + m gridDim.x); a
    // warp's first chunk of a sweep is its own number, the next ones come
    // from the counter (warp-uniform).
    auto slot0 = [&](unsigned int m) -> unsigned int { return (blockIdx.x + m * gridDim.x) * 32; };
    const unsigned int stride = n_warps * gridDim.x * 32;  // static mapping of the landing: chunks warp, warp + n_warps, ...
    auto grab = [&]() -> unsigned int {
        unsigned int m = 0;
        if (lane == 0) m = atomicAdd(&s_next, 1);
        return n_warps + __shfl_sync(0xffffffffu, m, 0);
    };
    const double ie = P.inv_eps, mie = P.mie;
    const long long W = P.W;
    int cyc = 0;
    int K = 0;
    __shared__ int s_miss;
    const bool band_ok = mode == MODE_ETD && !T_known && P.band_m > 0;

    // attempt 1 replays the window with every trajectory row when a landing
    // row fell outside the band of attempt 0
    for (int attempt = 0;; ++attempt) {
    const bool band = band_ok && attempt == 0;
    for (unsigned int m = warp; m < my_chunks; m += n_warps) {
        const unsigned int i = slot0(m) + lane;
        int2 tr = make_int2(0, 0);
        if (i < n && !fine_only) {
            if (T_known) {
                Track s;
                s.flags = 0;
                track_resolve(s, P, Tin[i]);
                B.T[i] = s.T;
                B.o[i] = s.o;
                B.N[i] = s.N;
                tr = make_int2(s.flags, s.need);
            } else if (band) {
                tr.x = band_bits(P, B.T[i]);
            }
            B.tr[i] = tr;
        }
        if (STAGE == STAGE_RESIDENT) {
            stage[m].y[lane] = i < n ? B.y[i] : make_double2(0.0, 0.0);
            stage[m].tr[lane] = tr;
        }
    }

    __syncthreads();
    // half-steps: sweep A(k), cycle, sweep B(k), cycle (one copy of the cycle's code)
    for (int hs = 0;; ++hs) {
        const int k = hs >> 1;
        if (!(hs & 1)) {
        // ---- sweep A(k): finish step k-1, sample k, deposit stage pair 1 of step k
        const bool last_fine = fine_only && k == n_fine;
        const bool k0 = k == 0;
        unsigned int cnt = 0;
        int cur = 0;
        unsigned int m = warp;
        if (STAGE == STAGE_NEXT) {
            if (m < my_chunks && slot0(m) + lane < n) prefetch_chunk<SOLVER>(B, slot0(m) + lane, true, fine_only, k0, my_stage, lane);
            cp_async_commit();
        }
        // warp-uniform trip count: lanes past the end run with an empty cell
        for (; m < my_chunks; cur ^= 1) {
            const unsigned int mn = grab();
            const unsigned int i = slot0(m) + lane;
            const bool valid = i < n;
            Stage<SOLVER>* const S = stage + m;  // STAGE_RESIDENT
            ChunkIn in;
            if (STAGE == STAGE_NEXT) {
                if (mn < my_chunks && slot0(mn) + lane < n) prefetch_chunk<SOLVER>(B, slot0(mn) + lane, true, fine_only, k0, my_stage + (cur ^ 1), lane);
                cp_async_commit();
                cp_async_wait<1>();
                in = read_stage<SOLVER>(my_stage + cur, lane);
            } else if (STAGE == STAGE_RESIDENT) {
                in = read_stage<SOLVER>(S, lane);
            } else if (valid) {
                in = load_chunk<SOLVER>(B, i, true, fine_only, k0);
            }
            m = mn;
            double R = valid ? in.y.x : 0.0, V = valid ? in.y.y : 0.0;
            if (!valid) {
            } else if (k > 0) {
                const double ea = mesh_gather(tab, s_cyc.edges[0], s_cyc.edges[1], in.cj.x, in.ca.x);
                const double eb = mesh_gather(tab + Np1, s_cyc.edges[2], s_cyc.edges[3], in.cj.y, in.ca.y);
                double Rn, Vn;
                if (SOLVER == 1) {
                    // ce = (e1, e3), ea = e2, eb = e4, cx.x = (Phi_h y)_R
                    const double e1 = in.ce.x, e3 = in.ce.y;
                    const double Bv = fma(P.c1, V, -dmul_i(P.imul, P.s1, R));
                    const double e23 = ea + e3;
                    Rn = fma(P.h6, fma(P.tsh, e23, dmul_i(P.imul, P.s1, e1)), in.cx.x);
                    Vn = fma(P.h6, fma(P.tch, e23, fma(P.c1, e1, eb)), Bv);
                } else {
                    // ce = partial sums, cx = (R3, R4), ea = e3, eb = e4
                    const double k3V = fma(mie, in.cx.x, ea);
                    const double V4 = fma(P.h, k3V, V);
                    const double k4R = ie * V4, k4V = fma(mie, in.cx.y, eb);
                    const double sR = in.ce.x + k4R;
                    const double sV = (in.ce.y + 2.0 * k3V) + k4V;
                    Rn = fma(P.h6, sR, R);
                    Vn = fma(P.h6, sV, V);
                }
                if (!fine_only) {
                    int2 tr = in.tr;
                    // the sample is stored before tracking: a pending root at
                    // sample k+1 reads it back
                    if (!((tr.x & F_RES) && (detect_only || k > tr.y)) && (!band || band_holds(tr.x, k, P.band_m)))
                        __stcs(&B.traj[(size_t)k * n + i], make_double2(Rn, Vn));
                    const bool done = track_update(P, B, i, k, V, Vn, detect_only, tr);
                    if (STAGE == STAGE_RESIDENT) S->tr[lane] = tr;
                    cnt += done ? 0u : 1u;
                }
                R = Rn;
                V = Vn;
                if (STAGE == STAGE_RESIDENT) S->y[lane] = make_double2(R, V);
                if (STAGE != STAGE_RESIDENT || last_fine) B.y[i] = make_double2(R, V);
            } else if (!fine_only) {
                __stcs(&B.traj[i], make_double2(R, V));
                cnt += 1u;
            }
            if (last_fine) continue;
            // stage pair 1
            Cell ca, cb;
            double2 cx;
            if (SOLVER == 1) {
                ca = mesh_locate<POW2>(P, R);                            // stage 1: y
                cb = mesh_locate<POW2>(P, fma(P.sh, V, dmul_i(P.imul, P.ch, R)));  // stage 3: Phi_h/2 y
                cx = make_double2(fma(P.s1, V, dmul_i(P.imul, P.c1, R)), 0.0);  // (Phi_h y)_R
            } else {
                ca = mesh_locate<POW2>(P, R);                            // stage 1: y
                const double R2 = fma(P.h2, ie * V, R);                  // stage 2: y + h/2 k1
                cb = mesh_locate<POW2>(P, R2);
                cx = make_double2(R2, 0.0);
            }
            if (!valid) ca.j = cb.j = -3;
            deposit_cell<HIST>(my_hist, Np1, ca, W);
            deposit_cell<HIST>(my_hist + words, Np1, cb, W);
            if (STAGE == STAGE_RESIDENT) {
                S->ca[lane] = make_double2(ca.a, cb.a);
                S->cj[lane] = make_short2((short)ca.j, (short)cb.j);
                if constexpr (SOLVER == 1) S->cx[lane] = cx.x;
                else S->cx[lane] = cx;
            } else if (valid) {
                B.ca[i] = make_double2(ca.a, cb.a);
                B.cj[i] = make_short2((short)ca.j, (short)cb.j);
                if (SOLVER == 1) B.cxr[i] = cx.x;
                else B.cx[i] = cx;
            }
        }
        if (STAGE == STAGE_NEXT) cp_async_wait<0>();
        if (last_fine) break;
        if (!fine_only) {
            cnt = __reduce_add_sync(0xffffffffu, cnt);
            if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(&s_cnt, (int)cnt);
        }
        } else {
        // ---- sweep B(k): gather pair 1, deposit stage pair 2
        int cur = 0;
        unsigned int m = warp;
        if (STAGE == STAGE_NEXT) {
            if (m < my_chunks && slot0(m) + lane < n) prefetch_chunk<SOLVER>(B, slot0(m) + lane, false, fine_only, false, my_stage, lane);
            cp_async_commit();
        }
        for (; m < my_chunks; cur ^= 1) {
            const unsigned int mn = grab();
            const unsigned int i = slot0(m) + lane;
            const bool valid = i < n;
            Stage<SOLVER>* const S = stage + m;  // STAGE_RESIDENT
            ChunkIn in;
            if (STAGE == STAGE_NEXT) {
                if (mn < my_chunks && slot0(mn) + lane < n) prefetch_chunk<SOLVER>(B, slot0(mn) + lane, false, fine_only, false, my_stage + (cur ^ 1), lane);
                cp_async_commit();
                cp_async_wait<1>();
                in = read_stage<SOLVER>(my_stage + cur, lane);
            } else if (STAGE == STAGE_RESIDENT) {
                in = read_stage<SOLVER>(S, lane);
            } else if (valid) {
                in = load_chunk<SOLVER>(B, i, false, fine_only, false);
            }
            m = mn;
            if (!valid) {
                in.y = make_double2(0.0, 0.0);
                in.ca = make_double2(0.0, 0.0);
                in.cx = make_double2(0.0, 0.0);
                in.cj = make_short2(-3, -3);
            }
            const double R = in.y.x, V = in.y.y;
            const double ea = mesh_gather(tab, s_cyc.edges[0], s_cyc.edges[1], in.cj.x, in.ca.x);
            const double eb = mesh_gather(tab + Np1, s_cyc.edges[2], s_cyc.edges[3], in.cj.y, in.ca.y);
            double Pa, Pb;
            if (SOLVER == 1) {
                // ea = e1 at y, eb = e3 at Phi_h/2 y
                Pa = fma(P.sh, fma(P.h2, ea, V), P.ch * R);              // stage 2
                Pb = fma(P.hsh, eb, in.cx.x);                            // stage 4
                if (STAGE == STAGE_RESIDENT) S->ce[lane] = make_double2(ea, eb);
                else if (valid) B.ce[i] = make_double2(ea, eb);
            } else {
                // ea = e1 at y, eb = e2 at y + h/2 k1, cx.x = R2
                const double k1R = ie * V, k1V = fma(mie, R, ea);
                const double V2 = fma(P.h2, k1V, V);
                const double k2R = ie * V2, k2V = fma(mie, in.cx.x, eb);
                const double R3 = fma(P.h2, k2R, R), V3 = fma(P.h2, k2V, V);
                const double k3R = ie * V3;
                const double R4 = fma(P.h, k3R, R);
                Pa = R3;                                                 // stage 3
                Pb = R4;                                                 // stage 4
                const double2 part = make_double2((k1R + 2.0 * k2R) + 2.0 * k3R, k1V + 2.0 * k2V);
                if constexpr (STAGE == STAGE_RESIDENT && SOLVER == 0) {
                    S->ce[lane] = part;
                    S->cx[lane] = make_double2(R3, R4);
                } else if (valid) {
                    B.ce[i] = part;
                    B.cx[i] = make_double2(R3, R4);
                }
            }
            Cell ca2 = mesh_locate<POW2>(P, Pa), cb2 = mesh_locate<POW2>(P, Pb);
            if (!valid) ca2.j = cb2.j = -3;
            deposit_cell<HIST>(my_hist, Np1, ca2, W);
            deposit_cell<HIST>(my_hist + words, Np1, cb2, W);
            if (STAGE == STAGE_RESIDENT) {
                S->ca[lane] = make_double2(ca2.a, cb2.a);
                S->cj[lane] = make_short2((short)ca2.j, (short)cb2.j);
            } else if (valid) {
                B.ca[i] = make_double2(ca2.a, cb2.a);
                B.cj[i] = make_short2((short)ca2.j, (short)cb2.j);
            }
        }
        if (STAGE == STAGE_NEXT) cp_async_wait<0>();
        }
        const bool control = !(hs & 1) && !fine_only;
        if (!field_cycle<HIST>(cyc++, control)) return;
        if (control && s_stop) {
            K = k;
            break;
        }
    }

    if (blockIdx.x == 0 && threadIdx.x == 0 && !fine_only) *B.K_out = K;
    if (detect_only) {
        // step 1 alone leaves y^n as it was: it is row 0 of the trajectory
        for (unsigned int i = slot0(warp) + lane; i < n; i += stride) B.y[i] = B.traj[i];
        return;
    }
    if (mode != MODE_ETD) return;

    // ---- landing (step 3) and extrapolation (step 4); with the band, a
    // particle whose landing rows were not all stored marks a miss
    bool miss = false;
    for (unsigned int i = slot0(warp) + lane; i < n; i += stride) {
        const double o = B.o[i], T = B.T[i];
        const int N = B.N[i];
        const int nt = N > 0 ? 2 : 1;
        if (band) {
            const int x = B.tr[i].x;
            bool held = true;
            for (int t = 0; t < nt; ++t) {
                const int kk = (int)floor(t == 0 ? o : o + T);
                held = held && band_holds(x, kk, P.band_m) && band_holds(x, kk + 1, P.band_m) &&
                       band_holds(x, kk + 2, P.band_m);
            }
            if (!held) {
                miss = true;
                continue;
            }
        }
        double y[2][2];
        for (int t = 0; t < nt; ++t) {
            const double u = t == 0 ? o : o + T;
            const int kk = (int)floor(u);
            const double sf = u - (double)kk;
            const double2 a = B.traj[(size_t)kk * n + i];
            const double2 b = B.traj[(size_t)(kk + 1) * n + i];
            const double2 cc = B.traj[(size_t)(kk + 2) * n + i];
            y[t][0] = interp3(a.x, b.x, cc.x, sf);
            y[t][1] = interp3(a.y, b.y, cc.y, sf);
        }
        B.y[i] = make_double2(extrapolate(y[0][0], y[nt - 1][0], N), extrapolate(y[0][1], y[nt - 1][1], N));
    }
    if (!band) return;
    if (__syncthreads_or(miss) && threadIdx.x == 0) atomicOr(&B.notdone[3], 1);
    if (!grid_sync()) return;
    if (threadIdx.x == 0) s_miss = ld_acquire_s32(&B.notdone[3]);
    __syncthreads();
    if (!s_miss) return;
    // replay from y^n (row 0) with every row, for every particle
    for (unsigned int i = slot0(warp) + lane; i < n; i += stride) B.y[i] = B.traj[i];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        atomicAdd(&B.notdone[4], 1);
    }
    K = 0;
    if (!grid_sync()) return;
    }
}

}  // namespace pic
