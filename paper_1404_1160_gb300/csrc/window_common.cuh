// window_common.cuh -- device pieces shared by the FP64 and FP32 window
// kernels: the block-wide int64 scan of the charge, the bounded grid barrier
// and the cp.async helpers.  Everything is static/inline, so each
// translation unit keeps its own copy.
#pragma once

#include "pic_internal.h"

namespace pic {

static __device__ __forceinline__ long long warp_incl_scan64(long long x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    return x;
}

// For both fields f = 0, 1: g_j = sum_{m<j} (q_m + q_{m+1}), j = 0..Nc
// (block-wide exclusive scans in shared memory, done together).
static __device__ void block_exscan_pairs2(const long long* q, long long* g, int Nc, long long* s_warp) {
    const int T = blockDim.x, t = threadIdx.x, lane = t & 31, w = t >> 5, nw = T >> 5;
    const int Np1 = Nc + 1;
    const int per = (Nc + T - 1) / T;
    const int beg = min(t * per, Nc), end = min(beg + per, Nc);
    long long s0 = 0, s1 = 0;
    for (int m = beg; m < end; ++m) {
        s0 += q[m] + q[m + 1];
        s1 += q[Np1 + m] + q[Np1 + m + 1];
    }
    const long long x0 = warp_incl_scan64(s0), x1 = warp_incl_scan64(s1);
    if (lane == 31) {
        s_warp[w] = x0;
        s_warp[32 + w] = x1;
    }
    __syncthreads();
    if (w == 0) {
        long long y0 = (lane < nw) ? s_warp[lane] : 0, y1 = (lane < nw) ? s_warp[32 + lane] : 0;
        y0 = warp_incl_scan64(y0);
        y1 = warp_incl_scan64(y1);
        if (lane < nw) {
            s_warp[lane] = y0;
            s_warp[32 + lane] = y1;
        }
    }
    __syncthreads();
    long long r0 = x0 - s0 + (w > 0 ? s_warp[w - 1] : 0);
    long long r1 = x1 - s1 + (w > 0 ? s_warp[32 + w - 1] : 0);
    for (int m = beg; m < end; ++m) {
        g[m] = r0;
        g[Np1 + m] = r1;
        r0 += q[m] + q[m + 1];
        r1 += q[Np1 + m] + q[Np1 + m + 1];
    }
    if (end == Nc && beg < end) {
        g[Nc] = r0;
        g[Np1 + Nc] = r1;
    }
    __syncthreads();
}

// ---------------------------------------------------------- field cycle
//
// Every block adds its charge of a cycle to the cycle's global words and
// needs the sum over all blocks.  Where the node charge leaves room
// (P.q_cb > 0), the words count their own arrivals: a block adds
// (v << q_cb) + 1 to EVERY word of the slot, and a reader takes a word as
// complete when it has grown by n_blocks (mod 2^q_cb) since the slot's last
// use.  The growth is then exactly (Q << q_cb) + n_blocks, so the words are
// never cleared; each block keeps the last complete value of every word
// (`prev`, the same in all blocks).  No fence, arrival counter or barrier
// lies between the adds and the reads, and nothing but the words themselves
// passes between blocks, so relaxed accesses suffice.  Two slots alternate:
// a block adds to a slot again only after it has seen the cycle in between
// complete, which every block joins only after it has read the slot.
// The cycle is bound by L2 round trips (~1 k clocks each); the release
// counter, the polling barrier and the charge load that it replaces took
// three more of them (and still serve n W too large for the count and meshes
// beyond the register build).  One macro step, GB300, with the packed words
// and the single-barrier build below: FP32 10^6 particles, 256 cells 4.26 ->
// 4.04 ms; a 12-beam batch 6.90 -> 5.71 ms; FP64 10^6 9.65 -> 9.51 ms; two FP64
// steps of 20000 particles 10.3 -> 9.17 ms.

// What the end of a sweep needs, in shared memory: the field cycle is a
// function of its own (out of line, so that its registers do not add to the
// sweeps'), and it reads its parameters from here.
struct CycleCtx {
    unsigned long long* Qring;   // kQSlots slots of charge words
    unsigned int* bar;           // grid barrier (barrier form)
    int* status;
    long long wait_ns, W;
    double q_unit, q_half, inv_hr, invW;
    float q_half_f;
    int n_cells, c, log2W, parity_odd;
    int copies;                  // histogram copies
    int hs_a, hs_b;              // FP32 form: split of the right weights
    int q_cb;                    // count bits of the words; 0: barrier form
    int n_blocks, expect, lb;    // blocks that share the words, arrivals of one use, this block's index
    int hist, tabA, tabB, g, node_c;  // byte offsets in the dynamic shared memory
    double edges[4];             // FP64: rE at the mesh edges of both fields; FP32: 4 floats for each stage pair
};
static __shared__ CycleCtx s_cyc;
static __device__ __forceinline__ float* edges32(int pair) { return (float*)s_cyc.edges + 4 * pair; }
static __shared__ long long s_tot[64];
static __shared__ unsigned int s_gen;                    // generation of the grid barrier
static __shared__ int s_ok, s_cnt, s_next, s_stop;       // wait state, not-done count, next unit of a sweep, all done
extern __shared__ __align__(16) unsigned char smem_raw[];

// Thread 0 fills s_cyc at kernel start (the caller's block barrier follows).
static __device__ __forceinline__ void cycle_setup(const DevParams& P, unsigned long long* Qring, unsigned int* bar,
                                                   int* status, int n_blocks, int lb, int hist, int tabA, int tabB,
                                                   int g, int node_c) {
    if (threadIdx.x != 0) return;
    s_cyc.Qring = Qring;
    s_cyc.bar = bar;
    s_cyc.status = status;
    s_cyc.wait_ns = P.wait_ns;
    s_cyc.W = P.W;
    s_cyc.q_unit = P.q_unit;
    s_cyc.q_half = P.q_half;
    s_cyc.inv_hr = P.inv_hr;
    s_cyc.invW = P.invW;
    s_cyc.q_half_f = P.q_half_f;
    s_cyc.n_cells = P.n_cells;
    s_cyc.c = P.c;
    s_cyc.log2W = P.log2W;
    s_cyc.parity_odd = P.parity_odd;
    s_cyc.copies = P.hist_copies;
    s_cyc.hs_a = P.hs_a;
    s_cyc.hs_b = P.hs_b;
    s_cyc.q_cb = P.q_cb;
    s_cyc.n_blocks = n_blocks;
    s_cyc.expect = n_blocks + P.bar_extra;
    s_cyc.lb = lb;
    s_cyc.hist = hist;
    s_cyc.tabA = tabA;
    s_cyc.tabB = tabB;
    s_cyc.g = g;
    s_cyc.node_c = node_c;
    s_gen = 0;
    s_ok = 1;
    s_cnt = 0;
    s_next = 0;
    s_stop = 0;
}

// Called on every 32nd spin of a polling loop; t0 is the time of the first
// call (0 before).  -1: give up (another block failed, or the time limit has
// passed), else the new t0.
static __device__ __noinline__ long long wait_expired(int* status, long long wait_ns, long long t0) {
    if (ld_acquire_s32(status) != 0) return -1;
    const long long now = global_ns();
    if (t0 == 0) return now;
    if (now - t0 > wait_ns) {
        atomicCAS(status, 0, (int)DEV_TIMEOUT);
        return -1;
    }
    return t0;
}

// Growth of R consecutive charge words since the slot's last use, once they
// are complete: (Q_j << q_cb) + arrivals for nodes j0 .. j0 + R - 1 of the
// field at Qf (clamped to the last node; kept values at prev).
template <int R>
static __device__ __forceinline__ void poll_nodes(const unsigned long long* Qf, const unsigned long long* prev, int j0,
                                                  unsigned long long (&d)[R]) {
    const int Nc = s_cyc.n_cells;
    const unsigned int mask = (1u << s_cyc.q_cb) - 1u, expect = (unsigned int)s_cyc.expect;
    long long t0 = 0;
    unsigned spins = 0;
    for (;;) {
        bool done = true;
#pragma unroll
        for (int r = 0; r < R; ++r) d[r] = ld_relaxed_u64(Qf + q_node(min(j0 + r, Nc)));
#pragma unroll
        for (int r = 0; r < R; ++r) {
            d[r] -= prev[min(j0 + r, Nc)];
            done = done && ((unsigned int)d[r] & mask) == expect;
        }
        if (done) return;
        if ((++spins & 31) == 0 && (t0 = wait_expired(s_cyc.status, s_cyc.wait_ns, t0)) < 0) {
            s_ok = 0;
            return;
        }
    }
}

// Charge to field of one cycle for both fields, with the nodes in registers
// (one block barrier and no shared staging).  The first half of the block
// takes field 0, the second field 1; in warp w of a half, lane l < 31
// owns the R nodes j = (31 w + l) R + r, r < R, and lane 31 repeats the
// first nodes of the next warp, so that every lane finds E_{j+1} of its
// last node in the next lane.  q_j comes from the cycle's global charge;
// the exact trapezoid sums g_j = sum_{m<j} (q_m + q_{m+1}) are a warp scan
// plus the totals of the warps between the node's and the centre's (s_tot),
// S_j = g_j - g_c, and the node's field is field_at(j, S_j, q_j) (a struct of
// the form's own, passed to the lane below by shfl_next).  Each owned node goes
// to emit(f, j, field_j, field_{j+1}) (the latter unused at j = n_cells); after_scan()
// runs behind the block barrier, when every thread has passed its flush.
// Covers n_cells + 1 <= 31 R (blockDim/64) nodes.
// The last thread of the block also reads the control word (a count of
// particles not done) when `control`: s_stop = (count == 0).  Q: the slot;
// prev: its words when they were last complete (null: barrier form).
template <int R, class FieldAt, class Emit, class After>
static __device__ __forceinline__ bool field_build_regs_r(const unsigned long long* Q, unsigned long long* prev,
                                                          bool control, FieldAt field_at, Emit emit, After after_scan) {
    using Val = decltype(field_at(0, 0ll, 0ll));
    const int Nc = s_cyc.n_cells, Np1 = Nc + 1, c = s_cyc.c, cb = s_cyc.q_cb;
    const int H = blockDim.x >> 1;
    const int f = threadIdx.x >= H ? 1 : 0;
    const int u = threadIdx.x - f * H, lane = threadIdx.x & 31, w = u >> 5;
    const int j0 = (w * 31 + lane) * R;
    const unsigned long long* Qf = Q + (size_t)f * q_field_words(Nc);
    // warps whose first node lies beyond the mesh own no node (warp-uniform)
    const bool owns = w * 31 * R <= Nc;
    unsigned long long* const kept = prev + f * Np1;  // counted form
    long long q[R];
#pragma unroll
    for (int r = 0; r < R; ++r) q[r] = 0ll;
    if (owns) {
        if (prev) {
            unsigned long long d[R];
            poll_nodes<R>(Qf, kept, j0, d);
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (j0 + r <= Nc) q[r] = (long long)(d[r] >> cb);
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (j0 + r <= Nc) q[r] = (long long)__ldcg(Qf + q_node(j0 + r));
        }
    }
    if (control && threadIdx.x == blockDim.x - 1) {
        const unsigned long long* p = Q + 2 * q_field_words(Nc);
        if (prev) {
            unsigned long long d[1];
            poll_nodes<1>(p, prev + 2 * Np1, 0, d);
            s_stop = (d[0] >> cb) == 0ull;
            prev[2 * Np1] += d[0];
        } else {
            s_stop = __ldcg(p) == 0ull;
        }
    }
    long long g0 = 0;
    const int wc = c / (31 * R);  // the warp that owns the centre node
    if (owns) {
        const long long qn = __shfl_down_sync(0xffffffffu, q[0], 1);
        long long L = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long right = (r + 1 < R) ? q[(r + 1) % R] : qn;
            L += (j0 + r < Nc) ? q[r] + right : 0ll;
        }
        if (lane == 31) L = 0;  // its nodes belong to the next warp
        const long long incl = warp_incl_scan64(L);
        g0 = incl - L;
        if (lane == 31) s_tot[f * 32 + w] = incl;
        if (w == wc && lane != 31) {  // prefix of the centre node within its warp
            long long g = g0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (j0 + r == c) s_tot[f * 32 + 16] = g;
                if (r + 1 < R) g += (j0 + r < Nc) ? q[r] + q[(r + 1) % R] : 0ll;
            }
        }
    }
    __syncthreads();
    if (s_ok == 0) return false;
    after_scan();
    if (!owns) return true;
    if (prev && lane != 31) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (j0 + r <= Nc) kept[j0 + r] += ((unsigned long long)q[r] << cb) + (unsigned int)s_cyc.expect;
    }
    // totals of the warps between this one and the centre's (w, wc <= 15), by a butterfly
    long long t = 0;
    if (lane < w || lane < wc) {
        const long long x = s_tot[f * 32 + lane];
        t = (lane < w ? x : 0ll) - (lane < wc ? x : 0ll);
    }
#pragma unroll
    for (int d = 8; d >= 1; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
    t = __shfl_sync(0xffffffffu, t, 0);
    auto value = [&](int j, long long S, long long qj) -> Val { return field_at(min(j, Nc), S, qj); };
    long long S = g0 + t - s_tot[f * 32 + 16];
    Val Ecur = value(j0, S, q[0]);
    const Val En = shfl_next(Ecur);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int j = j0 + r;
        long long Sn = S;
        Val Enext = En;
        if (r + 1 < R) {
            Sn = S + ((j < Nc) ? q[r] + q[(r + 1) % R] : 0ll);
            Enext = value(j + 1, Sn, q[(r + 1) % R]);
        }
        if (lane != 31 && j <= Nc) emit(f, j, Ecur, Enext);
        Ecur = Enext;
        S = Sn;
    }
    return true;
}

template <class FieldAt, class Emit, class After>
static __device__ __forceinline__ bool field_build_regs(const unsigned long long* Q, unsigned long long* prev,
                                                        bool control, FieldAt field_at, Emit emit, After after_scan) {
    const int pp = 31 * (int)(blockDim.x >> 6), Np1 = s_cyc.n_cells + 1;  // nodes covered per node of a thread
    if (Np1 <= pp) return field_build_regs_r<1>(Q, prev, control, field_at, emit, after_scan);
    if (Np1 <= 2 * pp) return field_build_regs_r<2>(Q, prev, control, field_at, emit, after_scan);
    if (Np1 <= 3 * pp) return field_build_regs_r<3>(Q, prev, control, field_at, emit, after_scan);
    return field_build_regs_r<4>(Q, prev, control, field_at, emit, after_scan);
}

// Charge of every node into shared memory (q, 2 Np1), for meshes beyond the
// register form (barrier form of the cycle).
static __device__ __forceinline__ void stage_charge(const unsigned long long* Q, long long* q, bool control) {
    const int Nc = s_cyc.n_cells, Np1 = Nc + 1;
    for (int idx = threadIdx.x; idx < 2 * Np1; idx += blockDim.x) {
        const int f = idx >= Np1, j = idx - f * Np1;
        q[idx] = (long long)__ldcg(Q + (size_t)f * q_field_words(Nc) + q_node(j));
    }
    if (control && threadIdx.x == 0) s_stop = __ldcg(Q + 2 * q_field_words(Nc)) == 0ull;
}

// Adds this block's charge of every node, node(f, j), and with `control` its
// not-done count to a slot (see above).  Every lane of a warp calls node (the
// lanes hold consecutive nodes; past the end the last one).
template <class Node>
static __device__ __forceinline__ void flush_charge(unsigned long long* Q, bool control, Node node) {
    const int Nc = s_cyc.n_cells, Np1 = Nc + 1, cb = s_cyc.q_cb;
    for (int first = threadIdx.x & ~31; first < 2 * Np1; first += blockDim.x) {
        const int mine = first + (threadIdx.x & 31);
        const int idx = min(mine, 2 * Np1 - 1);
        const int f = idx >= Np1, j = idx - f * Np1;
        const unsigned long long v = node(f, j);
        if (mine != idx) continue;
        unsigned long long* w = Q + (size_t)f * q_field_words(Nc) + q_node(j);
        if (cb) atomicAdd(w, (v << cb) + 1ull);
        else if (v) atomicAdd(w, v);
    }
    if (control && threadIdx.x == blockDim.x - 1) {
        const unsigned long long v = (unsigned int)s_cnt;
        if (cb) atomicAdd(Q + 2 * q_field_words(Nc), (v << cb) + 1ull);
        else if (v) atomicAdd(Q + 2 * q_field_words(Nc), v);
    }
}

// Barrier form: clears the slot of the cycle after (one block does).
static __device__ __forceinline__ void clear_slot(unsigned long long* Q) {
    const int Nc = s_cyc.n_cells;
    for (int i = threadIdx.x; i < 2 * Nc + 3; i += blockDim.x) Q[q_used(Nc, i)] = 0ull;
}

// Barrier of the n_blocks blocks that share s_cyc.bar (the whole grid, or the
// blocks of one beam of a batch), with a time limit, in two halves so that
// a block can issue work that does not depend on the other blocks (loads of
// its own particles) between its arrival and its wait.
// Arrival: after the block's own barrier, one release reduction on the
// counter bar[0] (it orders every write the block made before it, the
// charge flush included, without waiting for a returned value).  Wait: one
// thread polls the counter with acquire loads until all n_blocks arrivals of
// this generation are in; the block barrier then passes the acquire on to
// the other threads.  The counter only grows within a launch (reset between
// launches), so generation g waits for g * n_blocks arrivals.
static __device__ __forceinline__ void grid_arrive() {
    __syncthreads();
    if (threadIdx.x == 0) {
        ++s_gen;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(s_cyc.bar) : "memory");
    }
}

// false if any block timed out or failed
static __device__ __forceinline__ bool grid_wait() {
    if (threadIdx.x == 0) {
        const unsigned int target = s_gen * (unsigned int)s_cyc.expect;
        long long t0 = 0;
        unsigned spins = 0;
        while ((int)(ld_acquire_u32(s_cyc.bar) - target) < 0) {
            if ((++spins & 31) == 0 && (t0 = wait_expired(s_cyc.status, s_cyc.wait_ns, t0)) < 0) {
                s_ok = 0;
                break;
            }
        }
    }
    __syncthreads();
    return s_ok != 0;
}

static __device__ __forceinline__ bool grid_sync() {
    grid_arrive();
    return grid_wait();
}

// The exchange of a cycle: flush, and in the barrier form the barrier.
// Returns the slot (null: a wait ran out) and the slot's kept words in *prev.
template <class Node>
static __device__ __forceinline__ unsigned long long* cycle_exchange(int cyc, bool control, unsigned long long** prev,
                                                                     Node node) {
    const int Nc = s_cyc.n_cells;
    const bool counted = s_cyc.q_cb > 0;
    unsigned long long* Q = s_cyc.Qring + (size_t)(counted ? cyc & 1 : cyc % 3) * q_slot_words(Nc);
    flush_charge(Q, control, node);
    if (counted) {
        *prev = (unsigned long long*)(smem_raw + s_cyc.g) + (cyc & 1) * (2 * (Nc + 1) + 1);
        return Q;
    }
    *prev = nullptr;
    if (s_cyc.lb == 0) clear_slot(s_cyc.Qring + (size_t)((cyc + 1) % 3) * q_slot_words(Nc));
    return grid_sync() ? Q : nullptr;
}

// ---- asynchronous copies global -> shared (cp.async, sm_80+)

static __device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned int d = (unsigned int)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem) : "memory");
}
static __device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
    const unsigned int d = (unsigned int)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(gmem) : "memory");
}
static __device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    const unsigned int d = (unsigned int)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gmem) : "memory");
}
static __device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
static __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

}  // namespace pic
