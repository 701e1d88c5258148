// window32.cu -- the FP32 form of the fine window of Algorithm ETDFSSModAlgo
// (Frenod, Hirstoaga & Lutz, Sec. 3): the same steps as window.cu (fine
// solver from y^n with period detection, quadratic landing at o and o+T,
// N-turn extrapolation), with the particle state and the push in binary32.
//
// Layout.  The state of fine step k of a window is the rotating-frame
// vector z_k = Phi(-t_k) y_k (see pic_device.cuh), stored as row k of a
// trajectory: row 0 is y^n itself (the public state, Phi(0) = I), rows
// 1..Kmax live in one array with a row stride of n rounded up to 128.  A
// step reads row k-1 and writes row k, so the trajectory the landing
// interpolates is the state the sweeps stream; the stage positions are
// recomputed from z when they are needed again, and the fields (e1, e3) of
// pair 1 are carried from the second sweep of a step to the first sweep of
// the next.  Per particle and fine step the window moves 8 B (read row k-1) +
// 4 B (tracking word) + 8 B (e1, e3) + 8 B (write row k) in the first sweep
// and 8 B (read row k) + 8 B (e1, e3) in the second.
//
// Field cycle (Poisson): as in the FP64 kernel, stages pair up (1,3) and
// (2,4); each pair is deposited by one sweep into per-block 32-bit
// histograms, flushed with 64-bit global atomics, and when all blocks have
// flushed every block turns the global int64 charge into its own field table
// of binary32 (E_j, E_{j+1} - E_j), computed in binary32 from the exact int64
// sums and per-node constants (field_cycle32).  Two tables are kept: the
// one of pair 1 (fields of R1, R3), read by the second sweep, and the one of
// pair 2 (R2, R4), read by the first sweep of the next step.
#include "pic_internal.h"
#include "window_common.cuh"

namespace pic {

constexpr int kW32Threads = 1024;
constexpr int kRowPad = 128;      // rows are padded to a multiple of this many slots
constexpr int kHist32CopiesMax = 4;  // histogram copies (lane l deposits into copy l mod copies)

// ---------------------------------------------------------------- deposit
//
// Block histogram of one field: per cell and copy four 32-bit words, the
// count C_j and the right weights qR in three parts summed separately,
// qR = h 2^a + m 2^b + l, so that S_j = H_j 2^a + M_j 2^b + L_j and the node
// charge is Q_j = W C_j - S_j + S_{j-1}, exactly.  hist32_split picks a and b
// so that no word overflows for the positions a block deposits into one copy.
// Every lane adds its own position with plain shared reductions: on this GPU
// that is several times faster than merging the lanes of a warp that share a
// cell first (match + reduce), and than 64-bit shared atomics.
//
// With W = 2^32 the weight of a position with x = (R - r_min)/h_r >= 1 is a
// multiple of 2^9, since x - floor(x) is a multiple of 2^-23: such a position
// (all but those in cell 0) takes its parts from the significand of 1 + f,
// with b = 9 and l = 0.  On a mesh of 256 cells or more f has 16 bits or
// fewer for most of the beam, so the middle part is 0 as well where h holds
// 16 bits (up to 65536 positions per copy) and two reductions remain of the
// four that a fixed 11/11/10-bit split with its count took.
__host__ __device__ constexpr long long hist32_positions_max() { return 1ll << 21; }

void hist32_split(DevParams* P, long long positions_per_block) {
    const long long M = (positions_per_block + P->hist_copies - 1) / P->hist_copies;
    int m = 0;
    while ((1ll << m) < M) ++m;
    const int s = m > 9 ? m - 9 : 0;  // bits of the middle part: M 2^(23 - s) <= 2^32
    if (m <= 20) {                    // M 2^s <= 2^32 too
        P->hs_a = 9 + s;
        P->hs_b = 9;
        P->hs_fast = P->log2W == 32 ? 1 : 0;
    } else {                          // 11/11/10 bits
        P->hs_a = 21;
        P->hs_b = 10;
        P->hs_fast = 0;
    }
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ float2 lds_f2(uint32_t a) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    return v;
}
// The sweeps' accesses to the histograms; block barriers separate them from
// the flush and the clearing, so no memory clobber is needed.
__device__ __forceinline__ void red_shared(uint32_t a, unsigned int v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(a), "r"(v));
}

// The histograms of a stage pair as the lanes of a warp see them: byte
// address of word w of cell j of this lane's copy = a (or b) + 4 jb + w plane,
// with jb = kFloorBits + j.  Layout: copies x 2 fields x 4 words x (n_cells +
// 1), so that the lanes of a warp meet different banks in different cells;
// n_cells + 1 is odd, so a cell's words lie 8, 16 and 24 banks on in the
// other copies.  (One 16-byte word per cell, four times fewer addresses, took
// 46.7 instead of 43.5 ms on 2 10^7 particles: a reduction then meets only
// every fourth bank.)
struct Hist32 {
    uint32_t a, b, plane;
    int hs_a, hs_b;
    unsigned int lim;   // fast form: bits(x) - bits(1) below this; 0: never
};
constexpr unsigned int kFloorBits = 0x4B000000u;  // bits of 2^23
constexpr unsigned int kOneBits = 0x3F800000u;    // bits of 1

// floor(x) as kFloorBits + j, and f = x - j (exact), for 0 <= x < 2^22: one
// add rounded down in place of a floor and a conversion on the slow pipe.
__device__ __forceinline__ unsigned int floor_bits(float x, float& f) {
    const float t = __fadd_rd(x, 8388608.0f);
    f = x - (t - 8388608.0f);
    return __float_as_uint(t);
}

// fast form (see above)
__device__ __forceinline__ void deposit32_fast(const Hist32& H, uint32_t base, float x) {
    float f;
    const unsigned int jb = floor_bits(x, f);
    const unsigned int g = __float_as_uint(1.0f + f);  // exact: 1 <= x, so f is a multiple of 2^-23
    const int s = H.hs_a - 9;
    const uint32_t c = base + (jb << 2);
    const unsigned int lo = g & ((1u << s) - 1u);
    red_shared(c, 1u);
    red_shared(c + H.plane, (g >> s) - (kOneBits >> s));
    if (lo) red_shared(c + 2 * H.plane, lo);
}

__device__ __forceinline__ void deposit32(const Hist32& H, uint32_t base, const Cell32& c) {
    if (c.j < 0) return;
    const uint32_t w = base + ((kFloorBits + (unsigned int)c.j) << 2);
    const unsigned int h = c.qR >> H.hs_a, m = (c.qR >> H.hs_b) & ((1u << (H.hs_a - H.hs_b)) - 1u),
                       l = c.qR & ((1u << H.hs_b) - 1u);
    red_shared(w, 1u);
    if (h) red_shared(w + H.plane, h);
    if (m) red_shared(w + 2 * H.plane, m);
    if (l) red_shared(w + 3 * H.plane, l);
}

// ------------------------------------------ located pairs, warp-uniform path
//
// Nearly every warp has all its positions on the mesh.  The pair helpers
// below test that once per pair of positions (one warp vote) and then run
// the cell arithmetic without the off-mesh selects, the gather without the
// edge division and the deposit in its fast form; a warp with a lane off the
// mesh (or at a NaN; for the deposits also in cell 0) runs the general
// locate32t / gather32 / deposit32.  Both give the same cells, weights,
// fields and sums.  Every lane of the warp must make the call.

// Fields at Ra (first table at ta, edges ed[0..1]) and Rb (second table tw
// bytes on, edges ed[2..3]).
__device__ __forceinline__ void locate_gather2(const DevParams& P, float Ra, float Rb, const float2* tab, int Np1,
                                               const float* ed, float& ea, float& eb) {
    const float xa = (Ra - P.r_min_f) * P.inv_hr_f, xb = (Rb - P.r_min_f) * P.inv_hr_f;
    const unsigned int lim = __float_as_uint(P.ncells_f);  // as unsigned, negatives and NaN lie above
    if (__all_sync(0xffffffffu, __float_as_uint(xa) < lim && __float_as_uint(xb) < lim)) {
        float fa, fb;
        const unsigned int ja = floor_bits(xa, fa), jb = floor_bits(xb, fb);
        const uint32_t t = smem_u32(tab) - (kFloorBits << 3);
        const float2 va = lds_f2(t + (ja << 3)), vb = lds_f2(t + 8u * (unsigned int)Np1 + (jb << 3));
        ea = fmaf(fa, va.y, va.x);
        eb = fmaf(fb, vb.y, vb.x);
    } else {
        const Cell32 ca = locate32t<false>(P, Ra), cb = locate32t<false>(P, Rb);
        ea = gather32(tab, ed[0], ed[1], ca);
        eb = gather32(tab + Np1, ed[2], ed[3], cb);
    }
}

// Deposits Ra into the first histogram and Rb into the second when `valid`.
__device__ __forceinline__ void locate_deposit2(const DevParams& P, const Hist32& H, float Ra, float Rb, bool valid) {
    const float xa = (Ra - P.r_min_f) * P.inv_hr_f, xb = (Rb - P.r_min_f) * P.inv_hr_f;
    if (__all_sync(0xffffffffu, __float_as_uint(xa) - kOneBits < H.lim && __float_as_uint(xb) - kOneBits < H.lim)) {
        if (valid) {
            deposit32_fast(H, H.a, xa);
            deposit32_fast(H, H.b, xb);
        }
    } else {
        const Cell32 ca = locate32(P, Ra), cb = locate32(P, Rb);
        if (valid) {
            deposit32(H, H.a, ca);
            deposit32(H, H.b, cb);
        }
    }
}

// Node charge Q_j = W C_j - S_j + S_{j-1} of one field from its histogram.  The
// lanes of a warp hold consecutive nodes, so S_{j-1} is the lane's below (the
// first lane reads it).  Every lane of the warp calls this.
__device__ __forceinline__ unsigned long long hist32_node(const unsigned int* h, int Np1, int j, int copies) {
    const int a = s_cyc.hs_a, b = s_cyc.hs_b;
    auto cell = [&](int m, unsigned int& C) -> unsigned long long {
        unsigned long long H = 0, M = 0, L = 0;
        for (int cp = 0; cp < copies; ++cp) {
            const unsigned int* w = h + cp * 8 * Np1 + m;
            C += w[0];
            H += w[Np1];
            M += w[2 * Np1];
            L += w[3 * Np1];
        }
        return (H << a) + (M << b) + L;
    };
    unsigned int C = 0, none = 0;
    const unsigned long long S = j < Np1 - 1 ? cell(j, C) : 0ull;
    unsigned long long Sm = __shfl_up_sync(0xffffffffu, S, 1);
    if (j == 0) Sm = 0ull;
    else if ((threadIdx.x & 31) == 0) Sm = cell(j - 1, none);
    return (unsigned long long)C * (unsigned long long)s_cyc.W - S + Sm;
}

// Field tables of one cycle from its global charge: exact int64 trapezoid
// sums S_j = g_j - g_c, then in binary32 E_j = float(S_j) cq_j with the
// per-node constant cq_j = q_unit / (2 r_j) (negated left of the axis for
// the odd reading) and E_c = float(Q_c) cq_c, cq_c = q_unit / h_r (0 for the
// odd reading); the table holds (E_j, E_{j+1} - E_j).  Each E_j is within
// 1.5 units in the last place of the exact node field, which the binary32
// bound of the form covers with a wide margin (a field error dE moves a
// particle by about h dE per stage).  All on the FP32 pipes: on this GPU the
// FP64 conversion of every node in every block was most of the build.  q is
// the int64 scan input (2 Np1), g the scan output, reused for E.
// `control`: the cycle carries the not-done count; s_stop = (count == 0).
// One call ends a sweep: the block's histograms into the cycle's words, the
// table of stage pair 1 (pair = 0) or 2 from the words of all blocks, and the
// histograms and the sweep's counters cleared for the next sweep.  false: a
// wait ran out of time.
static __device__ __forceinline__ void clear_hist32(unsigned int* hist, int words) {
    // 16-byte stores: the region starts aligned and holds a multiple of eight words
    for (int i = threadIdx.x; i < words / 4; i += blockDim.x) ((uint4*)hist)[i] = make_uint4(0u, 0u, 0u, 0u);
}
struct NodeField32 {
    float E, S;  // the field and float(S_j) (float(Q_c) at the centre)
};
static __device__ __forceinline__ NodeField32 shfl_next(const NodeField32& v) {
    return {__shfl_down_sync(0xffffffffu, v.E, 1), v.S};  // only E is used of the next lane's node
}

static __device__ __forceinline__ bool field_cycle32(int cyc, int pair, bool control) {
    __syncthreads();
    const int Nc = s_cyc.n_cells, Np1 = Nc + 1, c = s_cyc.c, copies = s_cyc.copies;
    unsigned int* hist = (unsigned int*)(smem_raw + s_cyc.hist);
    float2* tab = (float2*)(smem_raw + (pair ? s_cyc.tabB : s_cyc.tabA));
    float* edges = edges32(pair);
    const float* cq = (const float*)(smem_raw + s_cyc.node_c);
    unsigned long long* prev;
    const unsigned long long* Q = cycle_exchange(cyc, control, &prev, [&](int f, int j) {
        return hist32_node(hist + f * 4 * Np1, Np1, j, copies);
    });
    if (!Q) return false;
    auto clear = [&]() {
        clear_hist32(hist, copies * 8 * Np1);
        if (threadIdx.x == 0) {
            s_cnt = 0;
            s_next = 0;
        }
    };
    auto field_at = [&](int j, long long S, long long qj) -> NodeField32 {
        const float x = __ll2float_rn(j == c ? qj : S);
        return {x * cq[j], x};
    };
    auto edge = [&](int f, int j, float x) {
        // odd reading: the lower edge value carries the sign flip (rE / |R|)
        const float rE = x * s_cyc.q_half_f;
        if (j == 0) edges[2 * f] = s_cyc.parity_odd ? -rE : rE;
        if (j == Nc) edges[2 * f + 1] = rE;
    };
    if (field_in_regs(Nc, blockDim.x)) {
        auto emit = [&](int f, int j, const NodeField32& v, const NodeField32& next) {
            tab[f * Np1 + j] = make_float2(v.E, j < Nc ? next.E - v.E : 0.0f);
            edge(f, j, v.S);
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
    if (threadIdx.x < 2) {
        s_tot[threadIdx.x] = g[threadIdx.x * Np1 + c];
        s_tot[2 + threadIdx.x] = q[threadIdx.x * Np1 + c];
    }
    __syncthreads();
    float* e = (float*)g;  // E_idx in the slot of g[idx] (float 2 idx), which only this thread reads
    for (int idx = threadIdx.x; idx < 2 * Np1; idx += blockDim.x) {
        const int f = idx >= Np1, j = idx - f * Np1;
        const long long S = g[idx] - s_tot[f];
        const NodeField32 v = field_at(j, S, s_tot[2 + f]);
        edge(f, j, v.S);
        e[2 * idx] = v.E;
    }
    __syncthreads();
    clear();
    for (int idx = threadIdx.x; idx < 2 * Np1; idx += blockDim.x) {
        const int j = idx >= Np1 ? idx - Np1 : idx;
        tab[idx] = make_float2(e[2 * idx], j < Nc ? e[2 * idx + 2] - e[2 * idx] : 0.0f);
    }
    __syncthreads();
    return true;
}

// ------------------------------------------------------------ tracking

// Period tracking of one particle at sample k >= 1 (the FP32 twin of
// track_update in window_coop.cuh): a sign change of V between samples k-1
// and k is marked pending and counted as an extremum at sample k+1.  trw =
// flags | need << 8; until the period is known `need` holds the sample k_1
// before the first extremum.  Only the third extremum evaluates roots (with
// V_m = (Phi(t_m) z_m)_V of the stored rows) and resolves the period; that
// part, and the window cap, are out of line.
// Extremum times are kept as (integer, fraction).
static __device__ __noinline__ unsigned int track32_resolve(const DevParams& P, const WinBufs32& B, long long i, int k,
                                                           float Vold, float Vnew, bool detect_only,
                                                           unsigned int trw) {
    int flags = (int)(trw & 31u);
    int need = (int)(trw >> 8);
    auto V = [&](int m) -> float {
        const float2 z = m == 0 ? B.y[i] : B.traj[(size_t)(m - 1) * B.ld + i];
        const float2 cs = P.rot[rot_index(P, 2ll * m)];
        return rot_V(cs, z.x, z.y);
    };
    CTime T;
    T.i = P.spt;  // window cap without a third extremum: T = 2 pi eps
    T.f = 0.0f;
    if ((flags & F_NEXT) == 3) {
        const float s1 = quad_root01f(V(need), V(need + 1), V(need + 2));
        const float s3 = quad_root01f(V(k - 2), Vold, Vnew);
        T = ct_norm((long long)(k - 2) - need, s3 - s1);
    } else {
        flags |= F_FB;
    }
    if (detect_only) {
        flags |= F_RES;
        B.T[i] = T;
        need = 0;
    } else {
        const Decomp32 d = resolve32(P, T, true, flags);
        B.T[i] = d.T;
        B.o[i] = d.o;
        B.N[i] = d.N;
        need = d.need;
    }
    return (unsigned int)flags | ((unsigned int)need << 8);
}

// Returns true when the particle is done at sample k (resolved and every
// sample it needs is produced).
__device__ __forceinline__ bool track32_update(const DevParams& P, const WinBufs32& B, long long i, int k, float Vold,
                                               float Vnew, bool detect_only, unsigned int& trw) {
    if (!(trw & (unsigned int)F_RES)) {
        const bool pend = trw & (unsigned int)F_PEND, change = positive32(Vold) != positive32(Vnew);
        if (pend || change || k == P.Kmax) {
            if (pend) {
                trw += 1u - (unsigned int)F_PEND;
                if ((trw & 3u) == 1u) trw |= (unsigned int)(k - 2) << 8;
            }
            if ((trw & 3u) == 3u || k == P.Kmax) trw = track32_resolve(P, B, i, k, Vold, Vnew, detect_only, trw);
            else if (change) trw |= (unsigned int)F_PEND;
            B.tr[i] = trw;
        }
        if (!(trw & (unsigned int)F_RES)) return false;
    }
    return detect_only || k >= (int)(trw >> 8);
}

// ------------------------------------------------ cooperative Poisson window

// G consecutive slots of one lane: (R, V) or (e1, e3) pairs.
template <int G>
__device__ __forceinline__ void load_pairs(const float2* p, float (&v)[2 * G]) {
    if constexpr (G == 1) {
        const float2 a = *p;
        v[0] = a.x;
        v[1] = a.y;
    } else {
        const float4 a = *(const float4*)p;
        v[0] = a.x;
        v[1] = a.y;
        v[2] = a.z;
        v[3] = a.w;
    }
}
template <int G>
__device__ __forceinline__ void store_pairs(float2* p, const float (&v)[2 * G]) {
    if constexpr (G == 1) *p = make_float2(v[0], v[1]);
    else *(float4*)p = make_float4(v[0], v[1], v[2], v[3]);
}
template <int G>
__device__ __forceinline__ void load_words(const unsigned int* p, unsigned int (&v)[G]) {
    if constexpr (G == 1) {
        v[0] = *p;
    } else {
        static_assert(G == 2, "one or two slots per lane");
        const uint2 a = *(const uint2*)p;
        v[0] = a.x;
        v[1] = a.y;
    }
}

// What sweep A reads of a unit's slots of one lane.
template <int G>
struct UnitIn {
    float z[2 * G], e[2 * G];
    unsigned int tr[G];
};

// Shared memory of the FP32 window kernel (bytes).
static size_t coop32_smem_bytes(int n_cells, int copies, int block, bool kept) {
    const size_t Np1 = (size_t)n_cells + 1;
    return (size_t)copies * 8 * Np1 * sizeof(unsigned int)  // histograms; also the int64 scan input
           + 4 * Np1 * sizeof(float2)                     // tables of pair 1 and pair 2
           + cycle_words(n_cells, block, kept) * sizeof(long long)  // kept charge words, or scan output, then E
           + Np1 * sizeof(float);                         // field constants
}

// The window of one beam on blocks lb = 0..nb-1 of its own (the whole grid
// for a single beam, or a beam's share of a batch), G slots per lane and unit.
// AHEAD: the next unit's loads are issued before the current unit is worked on.
template <int G, bool AHEAD>
__device__ __forceinline__ void window32_coop_body(const DevParams& P, const WinBufs32& B, int mode, int T_known,
                                                   long long n_fine, const CTime* __restrict__ Tin, int lb, int nb) {
    constexpr unsigned int U = 32 * G;  // slots of a unit
    const int Nc = P.n_cells, Np1 = Nc + 1;
    const int copies = P.hist_copies;
    unsigned int* hist = (unsigned int*)smem_raw;    // copies x 2 fields x 4 words x Np1 cells
    float2* tabA = (float2*)(hist + copies * 8 * Np1);  // 2 Np1: fields of R1, R3
    float2* tabB = tabA + 2 * Np1;                   // 2 Np1: fields of R2, R4
    // scan output of the staged build (2 Np1), or the last complete charge
    // words of the two slots where the field is built in registers
    long long* g = (long long*)(tabB + 2 * Np1);
    unsigned long long* prev = (unsigned long long*)g;  // 2 x (2 Np1 + 1)
    float* cq = (float*)(g + cycle_words(Nc, blockDim.x, P.q_cb > 0));  // Np1
    if (P.q_cb)
        for (int i = threadIdx.x; i < 2 * (2 * Np1 + 1); i += blockDim.x) prev[i] = 0ull;
    clear_hist32(hist, copies * 8 * Np1);
    auto off = [&](const void* p) { return (int)((const unsigned char*)p - smem_raw); };
    cycle_setup(P, B.Qring, B.bar, B.status, nb, lb, off(hist), off(tabA), off(tabB), off(g), off(cq));
    for (int j = threadIdx.x; j < Np1; j += blockDim.x)
        cq[j] = (j == P.c) ? (P.parity_odd ? 0.0f : (float)(P.q_unit * P.inv_hr))
                           : (float)(((P.parity_odd && j < P.c) ? -P.q_half : P.q_half) / (P.r_min + (double)j * P.hr));

    const bool detect_only = mode == MODE_PERIODS, fine_only = mode == MODE_FINE, track = !fine_only;
    const unsigned int n = (unsigned int)P.n, ld = (unsigned int)B.ld;  // below 2^31
    const unsigned int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    // Work unit: U consecutive storage slots, lane l holding slots G l ..
    // G l + G - 1.  Block b owns the units u = b (mod grid); a warp's first
    // unit of a sweep is its own number, the next ones come from the counter,
    // in alternating directions from one sweep to the next so that the first
    // units a sweep reads are the last ones the previous sweep touched (still
    // in L2).
    const unsigned int n_units = ld / U;
    const unsigned int my_units = (unsigned int)lb < n_units ? (n_units - 1 - lb) / nb + 1 : 0;
    bool rev = false;
    auto grab = [&]() -> unsigned int {
        unsigned int m = 0;
        if (lane == 0) m = atomicAdd(&s_next, 1);
        return n_warps + __shfl_sync(0xffffffffu, m, 0);
    };
    auto base_of = [&](unsigned int m) -> unsigned int {
        return (lb + (rev ? my_units - 1 - m : m) * nb) * U + lane * G;
    };
    auto row = [&](unsigned int k) -> float2* {
        if (fine_only) return (k & 1) ? B.traj : B.y;
        return k == 0 ? B.y : B.traj + (size_t)(k - 1) * ld;
    };
    // Every slot is read and written by its own block only (set-up, sweeps and
    // landing alike): blocks exchange nothing but the charge words.
    const unsigned int my_slots = my_units * U;
    auto slot_of = [&](unsigned int s) -> unsigned int { return (lb + (s / U) * nb) * U + s % U; };

    if (!fine_only) {
        for (unsigned int s = threadIdx.x; s < my_slots; s += blockDim.x) {
            const unsigned int i = slot_of(s);
            if (i >= n) break;
            if (T_known) {
                int flags = 0;
                const Decomp32 d = resolve32(P, Tin[i], true, flags);
                B.T[i] = d.T;
                B.o[i] = d.o;
                B.N[i] = d.N;
                B.tr[i] = (unsigned int)flags | ((unsigned int)d.need << 8);
            } else {
                B.tr[i] = 0u;
            }
        }
    }

    int cyc = 0;
    int K = 0;
    // lane l deposits into copy l mod copies: the lanes of a warp hold
    // phase-space neighbours, which mostly fall into the same cell
    Hist32 H;
    H.a = smem_u32(hist + (lane & (copies - 1)) * 8 * Np1) - (kFloorBits << 2);
    H.b = H.a + 16u * (unsigned int)Np1;
    H.plane = 4u * (unsigned int)Np1;
    H.hs_a = P.hs_a;
    H.hs_b = P.hs_b;
    H.lim = P.hs_fast ? __float_as_uint(P.ncells_f) - kOneBits : 0u;
    __syncthreads();

    // half-steps: sweep A(k), cycle, sweep B(k), cycle (one copy of the cycle's code)
    for (int hs = 0;; ++hs) {
        const int k = hs >> 1;
        const float2 rb = P.rot[rot_index(P, 2ll * k)];      // Phi(t_k)
        const float2 rp = P.rot[rot_index(P, 2ll * k + 1)];  // Phi(t_k + h/2)
        if (!(hs & 1)) {
            // ---- sweep A(k): finish step k-1 (write row k), sample k, deposit stage pair 1 of step k
            const bool last_fine = fine_only && k == n_fine;
            float2 ra = rb, rm = rp;
            if (k > 0) {
                ra = P.rot[rot_index(P, 2ll * k - 2)];  // Phi(t_{k-1})
                rm = P.rot[rot_index(P, 2ll * k - 1)];  // Phi(t_{k-1} + h/2)
            }
            const float2* src = row(k > 0 ? k - 1 : 0);
            float2* dst = last_fine ? B.y : row(k);
            unsigned int cnt = 0;
            UnitIn<G> in;
            auto fetch = [&](unsigned int m) {
                const unsigned int b = base_of(m);
                load_pairs<G>(src + b, in.z);
                if (k > 0) load_pairs<G>(B.ce + b, in.e);
                if (track) load_words<G>(B.tr + b, in.tr);
            };
            unsigned int m = warp;
            if (AHEAD && m < my_units) fetch(m);
            while (m < my_units) {
                const unsigned int base = base_of(m);
                if (!AHEAD) fetch(m);
                UnitIn<G> cur = in;
                float(&z)[2 * G] = cur.z;
                float(&e)[2 * G] = cur.e;
                unsigned int(&tr)[G] = cur.tr;
                if (AHEAD) {
                    m = grab();
                    if (m < my_units) fetch(m);
                }
#pragma unroll
                for (int q = 0; q < G; ++q) {
                    const unsigned int i = base + q;
                    const bool valid = i < n;
                    float zR = z[2 * q], zV = z[2 * q + 1];
                    if (k > 0) {
                        const float R3 = rot_R(rm, zR, zV);
                        const float e1 = e[2 * q], e3 = e[2 * q + 1];
                        float e2, e4;
                        locate_gather2(P, lawson32_R2(P, R3, e1), lawson32_R4(P, rb, zR, zV, e3), tabB, Np1,
                                       edges32(1), e2, e4);
                        const float Vold = rot_V(ra, zR, zV);
                        lawson32_update(P, ra, rm, rb, e1, e2, e3, e4, zR, zV);
                        if (track && valid)
                            cnt += track32_update(P, B, i, k, Vold, rot_V(rb, zR, zV), detect_only, tr[q]) ? 0u : 1u;
                    } else if (track && valid) {
                        cnt += 1u;
                    }
                    if (last_fine) {
                        // the state leaves the rotating frame: y = Phi(t_k) z
                        z[2 * q] = rot_R(rb, zR, zV);
                        z[2 * q + 1] = rot_V(rb, zR, zV);
                        continue;
                    }
                    z[2 * q] = zR;
                    z[2 * q + 1] = zV;
                    // stage pair 1 of step k: R1 = (Phi(t_k) z)_R, R3 = (Phi(t_k + h/2) z)_R
                    locate_deposit2(P, H, rot_R(rb, zR, zV), rot_R(rp, zR, zV), valid);
                }
                if (k > 0) store_pairs<G>(dst + base, z);
                if (!AHEAD) m = grab();
            }
            rev = !rev;
            if (last_fine) break;
            if (track) {
                cnt = __reduce_add_sync(0xffffffffu, cnt);
                if (lane == 0 && cnt) atomicAdd(&s_cnt, (int)cnt);
            }
        } else {
            // ---- sweep B(k): gather pair 1 of step k, deposit stage pair 2
            const float2 rq = P.rot[rot_index(P, 2ll * k + 2)];  // Phi(t_k + h)
            const float2* srcB = row(k);
            float zn[2 * G];
            unsigned int m = warp;
            if (AHEAD && m < my_units) load_pairs<G>(srcB + base_of(m), zn);
            while (m < my_units) {
                const unsigned int base = base_of(m);
                float z[2 * G], e[2 * G];
                if (!AHEAD) load_pairs<G>(srcB + base, zn);
#pragma unroll
                for (int q = 0; q < 2 * G; ++q) z[q] = zn[q];
                if (AHEAD) {
                    m = grab();
                    if (m < my_units) load_pairs<G>(srcB + base_of(m), zn);
                }
#pragma unroll
                for (int q = 0; q < G; ++q) {
                    const bool valid = base + q < n;
                    const float zR = z[2 * q], zV = z[2 * q + 1];
                    const float R3 = rot_R(rp, zR, zV);
                    float e1, e3;
                    locate_gather2(P, rot_R(rb, zR, zV), R3, tabA, Np1, edges32(0), e1, e3);
                    e[2 * q] = e1;
                    e[2 * q + 1] = e3;
                    locate_deposit2(P, H, lawson32_R2(P, R3, e1), lawson32_R4(P, rq, zR, zV, e3), valid);
                }
                store_pairs<G>(B.ce + base, e);
                if (!AHEAD) m = grab();
            }
            rev = !rev;
        }
        const bool control = !(hs & 1) && track;
        if (!field_cycle32(cyc++, hs & 1, control)) return;
        if (control && s_stop) {
            K = k;
            break;
        }
    }

    if (lb == 0 && threadIdx.x == 0 && !fine_only) *B.K_out = K;
    if (mode != MODE_ETD) return;

    // ---- landing (step 3) and extrapolation (step 4); row k holds z_k
    for (unsigned int s = threadIdx.x; s < my_slots; s += blockDim.x) {
        const unsigned int i = slot_of(s);
        if (i >= n) break;
        const CTime o = B.o[i], T = B.T[i];
        const int N = B.N[i];
        float yv[2][2];
        const int nt = N > 0 ? 2 : 1;
        for (int t = 0; t < nt; ++t) {
            const CTime u = t == 0 ? o : ct_add(o, T);
            float R[3], V[3];
            for (int r = 0; r < 3; ++r) {
                const long long kk = (long long)u.i + r;
                const float2 z = row(kk)[i];
                const float2 cs = P.rot[rot_index(P, 2 * kk)];
                R[r] = rot_R(cs, z.x, z.y);
                V[r] = rot_V(cs, z.x, z.y);
            }
            yv[t][0] = interp3f(R[0], R[1], R[2], u.f);
            yv[t][1] = interp3f(V[0], V[1], V[2], u.f);
        }
        float2 out;
        if (N > 0) {
            const float Nf = (float)N;
            out = make_float2(fmaf(Nf, yv[1][0] - yv[0][0], yv[0][0]), fmaf(Nf, yv[1][1] - yv[0][1], yv[0][1]));
        } else {
            out = make_float2(yv[0][0], yv[0][1]);
        }
        B.y[i] = out;
    }
}

template <int G, bool AHEAD>
__global__ void __launch_bounds__(kW32Threads, 1) k_window32_coop(DevParams P, WinBufs32 B, int mode, int T_known,
                                                                  long long n_fine, const CTime* __restrict__ Tin) {
    window32_coop_body<G, AHEAD>(P, B, mode, T_known, n_fine, Tin, blockIdx.x, gridDim.x);
}

// ------------------------------------------- per-particle window (analytic E)

// The per-particle loops below keep the table position of fine step k,
// ia = 2k mod 2 spt, and advance it by one step with a compare instead of
// a remainder by the run-time table length (which costs more than the
// step's own arithmetic).  ia is even, so ia + 1 is always in the table.
__device__ __forceinline__ int rot_next(const DevParams& P, int ia) {
    const int t = ia + 2;
    return t == 2 * P.spt ? 0 : t;
}

// One fine step k -> k+1 of Lawson RK4 in the rotating frame, analytic
// field; ia = 2k mod 2 spt.
template <int FIELD>
__device__ __forceinline__ void step32_analytic(const DevParams& P, int ia, float& zR, float& zV) {
    const float2 a = P.rot[ia];
    const float2 m = P.rot[ia + 1];
    const float2 b = P.rot[rot_next(P, ia)];
    const float R3 = rot_R(m, zR, zV);
    const float e1 = field_analytic32(FIELD, rot_R(a, zR, zV));
    const float e3 = field_analytic32(FIELD, R3);
    const float e2 = field_analytic32(FIELD, lawson32_R2(P, R3, e1));
    const float e4 = field_analytic32(FIELD, lawson32_R4(P, b, zR, zV, e3));
    lawson32_update(P, a, m, b, e1, e2, e3, e4, zR, zV);
}

// y = Phi(t_k) z with ia = 2k mod 2 spt (y_at) or any k (y_of).
__device__ __forceinline__ float2 y_at(const DevParams& P, int ia, float zR, float zV) {
    const float2 cs = P.rot[ia];
    return make_float2(rot_R(cs, zR, zV), rot_V(cs, zR, zV));
}
__device__ __forceinline__ float2 y_of(const DevParams& P, long long k, float zR, float zV) {
    return y_at(P, rot_index(P, 2 * k), zR, zV);
}

template <int FIELD>
__device__ __forceinline__ void window32_local_body(const DevParams& P, const WinBufs32& B, int mode, int T_known,
                                                    long long n_iter, const CTime* __restrict__ Tin, int lb, int nb) {
    const long long n = P.n, ld = B.ld;
    const long long stride = (long long)nb * blockDim.x;
    int Kmax_seen = 0;
    for (long long i = (long long)lb * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float2 y0 = B.y[i];
        float zR = y0.x, zV = y0.y;
        if (mode == MODE_FINE) {
            int ia = 0;
            for (long long k = 0; k < n_iter; ++k) {
                step32_analytic<FIELD>(P, ia, zR, zV);
                ia = rot_next(P, ia);
            }
            B.y[i] = y_at(P, ia, zR, zV);
            continue;
        }
        if (mode == MODE_PERIODS) {
            int flags = 0;
            CTime t1, T;
            t1.i = 0;
            t1.f = 0.0f;
            T = t1;
            float vkm2 = 0.0f, vkm1 = zV;
            int K = 0, ia = 0;
            for (;;) {
                if (flags & F_RES) break;
                if (K == P.Kmax) {
                    flags |= F_FB | F_RES;
                    T.i = P.spt;
                    T.f = 0.0f;
                    break;
                }
                step32_analytic<FIELD>(P, ia, zR, zV);
                ia = rot_next(P, ia);
                ++K;
                const float v = y_at(P, ia, zR, zV).y;
                if (K >= 2 && positive32(vkm2) != positive32(vkm1)) {
                    const float s = quad_root01f(vkm2, vkm1, v);
                    const int ne = (flags & F_NEXT) + 1;
                    flags = (flags & ~F_NEXT) | (ne & F_NEXT);
                    if (ne == 1) {
                        t1.i = K - 2;
                        t1.f = s;
                    }
                    if (ne == 3) {
                        T = ct_norm((long long)(K - 2) - t1.i, s - t1.f);
                        flags |= F_RES;
                    }
                }
                vkm2 = vkm1;
                vkm1 = v;
            }
            B.T[i] = T;
            B.tr[i] = (unsigned int)flags;
            Kmax_seen = max(Kmax_seen, K);
            continue;
        }
        // MODE_ETD: n_iter macro steps of this particle
        int flags = 0;
        Decomp32 d;
        d.N = 0;
        d.need = 0;
        if (T_known) d = resolve32(P, Tin[i], true, flags);
        int K = 0;
        for (long long mstep = 0; mstep < n_iter; ++mstep) {
            float ya[2], yb[2];
            if (T_known) {
                // o, T and the stencils are known before the window starts
                const int k1 = d.o.i;
                const CTime u2 = ct_add(d.o, d.T);
                const int k2 = d.N > 0 ? u2.i : -10;
                float a[3], b[3], c[3], e[3];
                K = 0;
                int ia = 0;
                for (;;) {
                    const int r1 = K - k1, r2 = K - k2;
                    if (r1 >= 0 && r1 < 3) {
                        const float2 y = y_at(P, ia, zR, zV);
                        a[r1] = y.x;
                        b[r1] = y.y;
                    }
                    if (r2 >= 0 && r2 < 3) {
                        const float2 y = y_at(P, ia, zR, zV);
                        c[r2] = y.x;
                        e[r2] = y.y;
                    }
                    if (K >= d.need) break;
                    step32_analytic<FIELD>(P, ia, zR, zV);
                    ia = rot_next(P, ia);
                    ++K;
                }
                ya[0] = interp3f(a[0], a[1], a[2], d.o.f);
                ya[1] = interp3f(b[0], b[1], b[2], d.o.f);
                if (d.N > 0) {
                    yb[0] = interp3f(c[0], c[1], c[2], u2.f);
                    yb[1] = interp3f(e[0], e[1], e[2], u2.f);
                } else {
                    yb[0] = ya[0];
                    yb[1] = ya[1];
                }
            } else {
                // step 1 on the fly: track the extrema, store z_k as row k
                int fl = 0;
                CTime t1;
                t1.i = 0;
                t1.f = 0.0f;
                float vkm2 = 0.0f, vkm1 = zV;
                K = 0;
                int ia = 0;
                B.y[i] = make_float2(zR, zV);
                for (;;) {
                    if ((fl & F_RES) && K >= d.need) break;
                    if (K == P.Kmax) {
                        if (!(fl & F_RES)) {
                            CTime Tfb;
                            Tfb.i = P.spt;
                            Tfb.f = 0.0f;
                            fl |= F_FB;
                            d = resolve32(P, Tfb, true, fl);
                        }
                        break;
                    }
                    step32_analytic<FIELD>(P, ia, zR, zV);
                    ia = rot_next(P, ia);
                    ++K;
                    B.traj[(size_t)(K - 1) * ld + i] = make_float2(zR, zV);
                    const float v = y_at(P, ia, zR, zV).y;
                    if (!(fl & F_RES) && K >= 2 && positive32(vkm2) != positive32(vkm1)) {
                        const float s = quad_root01f(vkm2, vkm1, v);
                        const int ne = (fl & F_NEXT) + 1;
                        fl = (fl & ~F_NEXT) | (ne & F_NEXT);
                        if (ne == 1) {
                            t1.i = K - 2;
                            t1.f = s;
                        }
                        if (ne == 3) d = resolve32(P, ct_norm((long long)(K - 2) - t1.i, s - t1.f), true, fl);
                    }
                    vkm2 = vkm1;
                    vkm1 = v;
                }
                flags = fl;
                const int nt = d.N > 0 ? 2 : 1;
                for (int t = 0; t < nt; ++t) {
                    const CTime u = t == 0 ? d.o : ct_add(d.o, d.T);
                    float R[3], V[3];
                    for (int r = 0; r < 3; ++r) {
                        const long long kk = (long long)u.i + r;
                        const float2 z = kk == 0 ? B.y[i] : B.traj[(size_t)(kk - 1) * ld + i];
                        const float2 y = y_of(P, kk, z.x, z.y);
                        R[r] = y.x;
                        V[r] = y.y;
                    }
                    (t == 0 ? ya : yb)[0] = interp3f(R[0], R[1], R[2], u.f);
                    (t == 0 ? ya : yb)[1] = interp3f(V[0], V[1], V[2], u.f);
                }
                if (nt == 1) {
                    yb[0] = ya[0];
                    yb[1] = ya[1];
                }
            }
            if (d.N > 0) {
                const float Nf = (float)d.N;
                zR = fmaf(Nf, yb[0] - ya[0], ya[0]);
                zV = fmaf(Nf, yb[1] - ya[1], ya[1]);
            } else {
                zR = ya[0];
                zV = ya[1];
            }
            Kmax_seen = max(Kmax_seen, K);
        }
        B.y[i] = make_float2(zR, zV);
        if (n_iter > 0) {
            B.T[i] = d.T;
            B.o[i] = d.o;
            B.N[i] = d.N;
            B.tr[i] = (unsigned int)flags | ((unsigned int)d.need << 8);
        }
    }
    Kmax_seen = __reduce_max_sync(0xffffffffu, (unsigned)Kmax_seen);
    if ((threadIdx.x & 31) == 0 && Kmax_seen > 0) atomicMax((long long*)B.K_out, (long long)Kmax_seen);
}

template <int FIELD>
__global__ void __launch_bounds__(256) k_window32_local(DevParams P, WinBufs32 B, int mode, int T_known,
                                                        long long n_iter, const CTime* __restrict__ Tin) {
    window32_local_body<FIELD>(P, B, mode, T_known, n_iter, Tin, blockIdx.x, gridDim.x);
}

// ------------------------------------------------------------- batched form

constexpr int kBatchG = kWindow32Unit / 32;

// One cooperative launch advances every beam of a batch by one macro step:
// each block finds its beam, copies the beam's descriptor to shared memory
// and runs that beam's window on the beam's own blocks (its barriers count
// only them).  Beams never wait for each other.
__global__ void __launch_bounds__(kW32Threads, 1) k_window32_batch(const BeamDesc32* __restrict__ beams, int n_beams) {
    __shared__ BeamDesc32 D;
    __shared__ int s_beam;
    if (threadIdx.x == 0) {
        int lo = 0, hi = n_beams - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (beams[mid].first_block <= (int)blockIdx.x) lo = mid;
            else hi = mid - 1;
        }
        s_beam = lo;
    }
    __syncthreads();
    {
        const unsigned int* src = reinterpret_cast<const unsigned int*>(beams + s_beam);
        unsigned int* dst = reinterpret_cast<unsigned int*>(&D);
        for (int i = threadIdx.x; i < (int)(sizeof(BeamDesc32) / 4); i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    const int lb = (int)blockIdx.x - D.first_block;
    if (threadIdx.x == 0) atomicMin(&D.t_ns[0], (unsigned long long)global_ns());
    if (D.coop) window32_coop_body<kBatchG, false>(D.P, D.B, MODE_ETD, D.T_known, 0, D.Tin, lb, D.n_blocks);
    else if (D.P.field == 1) window32_local_body<1>(D.P, D.B, MODE_ETD, D.T_known, 1, D.Tin, lb, D.n_blocks);
    else window32_local_body<2>(D.P, D.B, MODE_ETD, D.T_known, 1, D.Tin, lb, D.n_blocks);
    __syncthreads();  // the block's last thread is done before its end time
    if (threadIdx.x == 0) atomicMax(&D.t_ns[1], (unsigned long long)global_ns());
}

__global__ void k_batch_reset(const BeamDesc32* __restrict__ beams, int n_beams) {
    const int b = blockIdx.x;
    if (b >= n_beams) return;
    const BeamDesc32& D = beams[b];
    if (D.coop) {
        const int Nc = D.P.n_cells;
        for (int s = 0; s < kQSlots; ++s)
            for (int i = threadIdx.x; i < 2 * Nc + 3; i += blockDim.x)
                D.B.Qring[s * q_slot_words(Nc) + q_used(Nc, i)] = 0ull;
        for (int i = threadIdx.x; i < 64; i += blockDim.x) D.B.bar[i] = 0u;
    }
    if (threadIdx.x == 0) {
        *D.B.K_out = 0;
        *D.B.status = 0;
        D.t_ns[0] = ~0ull;
        D.t_ns[1] = 0ull;
    }
}

__global__ void k_batch_status(const BeamDesc32* __restrict__ beams, int n_beams, int* __restrict__ out) {
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < n_beams; b += gridDim.x * blockDim.x)
        out[b] = *beams[b].B.status;
}

size_t window32_batch_smem(int max_cells, int copies, int block, bool kept) {
    return max_cells > 0 ? coop32_smem_bytes(max_cells, copies, block, kept) : 0;
}

cudaError_t window32_batch_open(size_t* most) { return open_shared_memory((const void*)k_window32_batch, most); }

cudaError_t window32_batch_occupancy(int block, size_t smem, int* blocks_per_sm) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_window32_batch, block, smem);
}

cudaError_t launch_window32_batch(const BeamDesc32* beams, int n_beams, int grid, int block, size_t smem,
                                  cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_window32_batch, beams, n_beams);
}

cudaError_t launch_batch_reset(const BeamDesc32* beams, int n_beams, cudaStream_t st) {
    k_batch_reset<<<n_beams, 256, 0, st>>>(beams, n_beams);
    return cudaGetLastError();
}

cudaError_t launch_batch_status(const BeamDesc32* beams, int n_beams, int* out, cudaStream_t st) {
    k_batch_status<<<1, 256, 0, st>>>(beams, n_beams, out);
    return cudaGetLastError();
}

// ------------------------------------------------------------- moments

// Per-block partial sums of the FP32 state, accumulated in FP64 (the global
// diagnostics of the form).
__global__ void k_moments32(DevParams P, WinBufs32 B, double* part_d, long long* part_i) {
    __shared__ double sd[32][kMomDoubles];
    __shared__ long long si[32][kMomInts];
    const long long n = P.n, stride = (long long)gridDim.x * blockDim.x;
    double a[kMomDoubles] = {0, 0, 0, 0, 0, 0, INFINITY, -INFINITY};
    long long b[kMomInts] = {LLONG_MAX, LLONG_MIN, 0};
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float2 y = B.y[i];
        const CTime Tc = B.T[i];
        const double R = y.x, V = y.y, T = (double)Tc.i + (double)Tc.f;
        const double R2 = R * R;
        a[0] += R;
        a[1] += V;
        a[2] += R2;
        a[3] += V * V;
        a[4] += R2 * R2;
        a[5] += T;
        a[6] = fmin(a[6], T);
        a[7] = fmax(a[7], T);
        const long long N = B.N[i];
        b[0] = min(b[0], N);
        b[1] = max(b[1], N);
        b[2] += (B.tr[i] & (unsigned int)F_FB) ? 1 : 0;
    }
    for (int d = 16; d >= 1; d >>= 1) {
        for (int q = 0; q < 6; ++q) a[q] += __shfl_xor_sync(0xffffffffu, a[q], d);
        a[6] = fmin(a[6], __shfl_xor_sync(0xffffffffu, a[6], d));
        a[7] = fmax(a[7], __shfl_xor_sync(0xffffffffu, a[7], d));
        b[0] = min(b[0], __shfl_xor_sync(0xffffffffu, b[0], d));
        b[1] = max(b[1], __shfl_xor_sync(0xffffffffu, b[1], d));
        b[2] += __shfl_xor_sync(0xffffffffu, b[2], d);
    }
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        for (int q = 0; q < kMomDoubles; ++q) sd[w][q] = a[q];
        for (int q = 0; q < kMomInts; ++q) si[w][q] = b[q];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int v = 1; v < nw; ++v) {
            for (int q = 0; q < 6; ++q) a[q] += sd[v][q];
            a[6] = fmin(a[6], sd[v][6]);
            a[7] = fmax(a[7], sd[v][7]);
            b[0] = min(b[0], si[v][0]);
            b[1] = max(b[1], si[v][1]);
            b[2] += si[v][2];
        }
        for (int q = 0; q < kMomDoubles; ++q) part_d[(size_t)blockIdx.x * kMomDoubles + q] = a[q];
        for (int q = 0; q < kMomInts; ++q) part_i[(size_t)blockIdx.x * kMomInts + q] = b[q];
    }
}

// ------------------------------------------------------------- launchers

// Work units of a sweep: how many slots a lane takes at once, and whether the
// next unit is loaded ahead.
enum Sweep32 { SWEEP_1 = 0, SWEEP_2 = 1, SWEEP_2_AHEAD = 2 };
static void* coop32_fn(int sweep) {
    if (sweep == SWEEP_1) return (void*)k_window32_coop<1, false>;
    return sweep == SWEEP_2 ? (void*)k_window32_coop<2, false> : (void*)k_window32_coop<2, true>;
}

cudaError_t window32_prepare(DevParams& P, int block, int blocks_per_sm, int sm_count, long long ld,
                             WindowLaunch* L) {
    L->coop_block = block;
    // Histogram copies (up to kHist32CopiesMax) relieve same-cell conflicts as
    // long as a block deposits at least 512 positions per copy and cycle; their
    // sums and clearing cost the cycle 2 n_cells words per copy, so copies x
    // n_cells stays within 2048.  Windows with 1 / 2 / 4 copies on GB300: 10^6 on
    // 256 cells 3.74 / 3.51 / 3.46 ms, 4 10^5 2.50 / 2.42 / 2.42, 1.5 10^5 1.90 /
    // 1.90 / 1.95; 2 10^6 on 1024 cells 6.77 / 6.76 / 7.45, 2 10^7 47.6 / 42.6 / 42.5.
    int copies = kHist32CopiesMax;
    const long long per_block_est = P.n / (sm_count > 0 ? sm_count : 1);
    while (copies > 1 && (coop32_smem_bytes(P.n_cells, copies, block, false) > 200 * 1024 ||
                          copies * P.n_cells > 2048 || per_block_est < 512ll * copies))
        copies >>= 1;
    P.hist_copies = copies;
    L->hist = 0;
    // One slot per lane while a warp has up to four such units (the tail of a
    // sweep is a unit, and a unit a chain of latencies); two beyond; and once
    // the 20 bytes per slot that a sweep reads outgrow half of L2 (64 MB),
    // loads one unit ahead.  Windows with SWEEP_1 / SWEEP_2 / SWEEP_2_AHEAD: 2 10^4
    // 1.82 / 2.01 / 2.07 ms, 4 10^5 2.42 / 2.52 / 2.58, 10^6 3.49 / 3.46 / 3.60, 2 10^6 (1024
    // cells) 7.14 / 6.76 / 6.78, 6 10^6 17.9 / 14.8 / 13.9, 2 10^7 55.4 / 42.6 / 38.9.
    const long long warps = (long long)sm_count * (block / 32);
    const int sweep = P.n <= 128 * warps ? SWEEP_1 : (20 * P.n <= (64ll << 20) ? SWEEP_2 : SWEEP_2_AHEAD);
    const int unit = sweep == SWEEP_1 ? 32 : 64;
    L->stage = sweep;
    size_t room = 0;
    cudaError_t e = open_shared_memory(coop32_fn(sweep), &room);
    if (e != cudaSuccess) return e;
    L->kept = field_in_regs(P.n_cells, block) && coop32_smem_bytes(P.n_cells, copies, block, true) <= room;
    L->coop_smem = coop32_smem_bytes(P.n_cells, copies, block, L->kept);
    if (L->coop_smem > room) return cudaErrorNotSupported;
    int bps = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, coop32_fn(sweep), block, L->coop_smem);
    if (e != cudaSuccess) return e;
    if (bps < 1) return cudaErrorInvalidConfiguration;
    const int want = blocks_per_sm > 0 ? blocks_per_sm : 1;
    if (want < bps) bps = want;
    const long long n_units = ld / unit;
    long long grid = (long long)bps * sm_count;
    // A unit for each of a block's first 16 warps before another block takes any: the
    // blocks of a small beam add to the same charge words, so fewer of them also
    // finish a cycle sooner, and other handles' windows run on the SMs they leave.
    // Units per block 1 / 4 / 8 / 16 / 32 in blocks of 512 threads on 256 cells: 2000
    // particles 1.30 / 1.31 / 1.32 / 1.36 / 1.54 ms, 2 10^4 1.38 / 1.38 / 1.34 / 1.36 / 1.53, 4 10^4 1.37 /
    // 1.37 / 1.37 / 1.36 / 1.52; of 1024 threads on 1024 cells: 2 10^4 2.50 / 2.49 / 2.34 / 2.35 / 2.41.
    const long long per = block / 32 < 16 ? block / 32 : 16;
    const long long blocks = (n_units + per - 1) / per;
    if (blocks < grid) grid = blocks < 1 ? 1 : blocks;
    L->coop_grid = (int)grid;
    // the 32-bit histogram words stay exact up to 2^21 positions per block,
    // field and cycle
    const long long per_block = (n_units + grid - 1) / grid * unit;
    if (per_block > hist32_positions_max()) return cudaErrorNotSupported;
    hist32_split(&P, per_block);
    return cudaSuccess;
}

long long window32_row_stride(long long n) { return (n + kRowPad - 1) / kRowPad * kRowPad; }

cudaError_t launch_window32_coop(const DevParams& P, const WinBufs32& B, const WindowLaunch& L, int mode,
                                 int T_known, long long n_fine, cudaStream_t st, long long* launches,
                                 const CTime* Tin) {
    DevParams Pc = P;
    Pc.q_cb = q_count_bits(P.n, P.W, (long long)L.coop_grid + P.bar_extra, L.kept);
    WinBufs32 Bc = B;
    void* args[] = {&Pc, &Bc, &mode, &T_known, &n_fine, &Tin};
    cudaError_t e = cudaLaunchCooperativeKernel(coop32_fn(L.stage), dim3(L.coop_grid), dim3(L.coop_block), args,
                                                L.coop_smem, st);
    if (launches) ++*launches;
    return e;
}

cudaError_t launch_window32_local(const DevParams& P, const WinBufs32& B, int mode, int T_known, long long n_iter,
                                  int block, int sm_count, cudaStream_t st, long long* launches, const CTime* Tin) {
    long long want = (P.n + block - 1) / block;
    long long cap = (long long)sm_count * 16;
    int grid = (int)(want < cap ? (want < 1 ? 1 : want) : cap);
    if (P.field == 1) k_window32_local<1><<<grid, block, 0, st>>>(P, B, mode, T_known, n_iter, Tin);
    else k_window32_local<2><<<grid, block, 0, st>>>(P, B, mode, T_known, n_iter, Tin);
    if (launches) ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_moments32(const DevParams& P, const WinBufs32& B, double* part_d, long long* part_i, int grid,
                             cudaStream_t st, long long* launches) {
    k_moments32<<<grid, 256, 0, st>>>(P, B, part_d, part_i);
    if (launches) ++*launches;
    return cudaGetLastError();
}

}  // namespace pic
