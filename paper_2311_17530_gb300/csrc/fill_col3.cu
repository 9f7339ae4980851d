// k = 3 column kernel: the fill of section 2 for three sequences, organised as a
// skewed register pipeline instead of independent tiles.
//
// Geometry (see c3:: in internal.h). A CTA owns the column (A, B): CTA rows
// rho = w*R + r (x0 = A*WR + rho) held by warp w in registers, lanes l
// (x1 = 32B + l), and it sweeps axis 2. At CTA time T lane l of warp w computes
// row r's cell at x2 = T - l - rho. Then, for the cell computed at time T+1,
//   e0  (x0-1)          is row rho-1 at time T        (same lane; warp above: ring)
//   e2  (x2-1)          is row rho   at time T        (same lane, same register)
//   e1  (x1-1)          is lane l-1 at time T         (shuffle at time T+1)
//   e01, e12            are lane l-1 at time T-1      (shuffled at time T)
//   e02                 is row rho-1 at time T-1
//   e012                is lane l-1, row rho-1 at time T-2 (shuffled at time T-1)
// so each step first finishes its own cells -- one fused add-max of a pre-reduced
// candidate P and the freshly shuffled e1 candidate, then the tag is cut off --
// and then prepares P for time T+1 and the e02/e012 pair D for time T+2 from
// values it already holds. Only the shuffle, that add-max and the cut sit on the
// step-to-step dependency chain.
//
// Keys. The kernel carries V = 8 H'(x) (the packed key of internal.h without its
// W part: the low three bits are zero) and adds to the candidate of move m a tag
// t(m), falling in m, so that one max finds the best value and, in its low three
// bits, the lowest mask among equals:
//     m    1 2 3 4 5 6 7
//     t(m) 7 5 4 3 2 1 0
// t(1) = 7 instead of 6 (no two moves share a tag, the order is the masks') makes
// t(1) - t(5) = t(3) + t(6) - t(7): with 7 on row -1's value, 4 on p01, 1 on p12
// and -5 on p02 every candidate gets its tag from a sum that is formed anyway,
// and e0 and e02 share vm + 7. Traceback bytes hold the tags; readers decode
// them (c3::mask_of_tag). Against keys with W in them (three instructions to
// recover the mask and rebuild the key) the cut is one, on the chain and off it.
//
// Pair scores never need an address in the step. p12 (row-independent, by lane
// and position) is looked up once per CTA by a staging warp, which fills a ring
// indexed by CTA time and lane; p02 (by row and position) by each warp for its own
// R rows, one block of steps ahead, into a ring indexed by tau = x2 + r, so that a
// lane reads its R rows of a step with R / 4 16-byte loads.
//
// Communication, all indexed by CTA time T (so every index inside an unrolled
// block of U steps is a compile-time offset):
//   ring[w][T]  row -1 of warp w at time T: (value, tag T) written by warp w-1
//               (its last row), or by the row staging warp for w = 0 (the
//               column above, face F0 at its time T + WR). A reader accepts an
//               entry when its tag is T, so warps never wait on a barrier.
//   f1r[T]      lane 0's inputs from the column to the left (its lane 31 at
//               time T + 31) and the corner from the column above-left, copied
//               by the column staging warp, which publishes how far it got.
//   F0, F1      global faces of this column, (value, tag) 8-byte entries whose
//               tag carries the launch epoch: no flags and no fences.
// A column runs CTA times -U .. nsteps - 1; the first block computes cells at
// x2 < 0 only, so that the candidates of time 0 and 1 are prepared like any
// other (their e0/e01/e02/e012 predecessors belong to the columns above and to
// the left). Traceback bytes and faces are stored from T = -U on (offset U).
//
// Cells outside the tensor are computed like any other. Positions x2 <= 0 take a
// sentinel code whose pair scores are kSentinelPair, and every value starts at
// kNeg, so such cells stay far below every valid key (the encode kernel's range
// check keeps that margin); the origin's pre-reduced candidate is set to
// H(0) = 0 when time 0 begins.
//
// Each lane stores its R traceback bytes of a step as one word, 32 * R contiguous
// bytes per warp step.
//
// What bounds it: the chain of columns. A step takes about 295 cycles (one warp per
// scheduler, 156 instructions, 80 of them on the half-rate integer pipe, 54 % of
// its cycles), a column starts about 56 steps after each of its producers (32 of
// them the skew, the rest the L2 round trip, the staging batch and the lag of the
// warps), and 528 columns of 152 at a time are 4,000 steps even at a lag of 32.
// Measured (ms, 700 x 760 x 800 / 128^3): 0.642 / 0.099, against 0.792 / 0.120 for
// the kernel with W in its keys, 8 warps of 4 rows, table addresses in the step and
// one staging warp. On the way: 4 rows x 8 warps 0.654 / 0.107; lane 31 storing
// face F1 itself, one entry pair at a time, 0.94 / 0.15; the shuffles of a step at
// its start instead of the step before, row -1 read when needed 0.96 / 0.145; two
// CTAs per SM 0.734 / 0.099 (each column's steps get slower, and the chain with
// them); staging batches of 8 / 4 rows on both axes 0.671 / 0.69; a 16-step block
// 1.06 (instruction fetch), 4-step groups 0.80; two steps per ring vote 0.70.
#include "api_internal.h"
#include "device_common.cuh"

#include <utility>

namespace msadp {

struct C3Smem {
    unsigned long long ring[c3::W][c3::SI][32];  // row -1 of warp w by CTA time: (value, tag)
    int32_t f1r[c3::SF + 1][c3::F1S];            // lane-0 inputs by CTA time: [3 + rho'], rho' = -1 .. WR-1
    int32_t p12r[c3::SP + c3::U][32];            // pair score (x1 of lane, x2) + 1 by x2 + lane, the first
                                                 // U rows again after the last
    int32_t p02r[c3::W][c3::R / 4][c3::SQ + c3::U][4];  // per warp: pair score (x0 of row r, x2) - 5 by r / 4,
                                                        // x2 + r and r mod 4, the first U slots again after the
                                                        // last (16-byte reads of consecutive slots: no conflict)
    int32_t f1b[c3::W][2][32];                   // per warp: lane 31's values of HF steps, twice
    int32_t prog[c3::W];                         // compute warp w has finished the steps < prog[w]
    int32_t staged;                              // f1r rows < staged hold this column's values
    int32_t failed;                              // a wait ran out: every warp leaves the column
    int32_t ctl[2];
    int32_t cur_prob;
    int32_t pad[3];
    int32_t corner[c3::R];                       // the far corner's lane's rows at the corner's CTA time
};

int col3_warps_per_cta() { return c3::W + 2; }

namespace {

__device__ __forceinline__ unsigned long long pack_entry(int value, int tag) {
    return (unsigned long long)(unsigned)value | ((unsigned long long)(unsigned)tag << 32);
}
__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long lds_u64_volatile(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.volatile.shared.u64 %0, [%1];" : "=l"(v) : "r"(smem_addr(p)));
    return v;
}
__device__ __forceinline__ int ld_acquire_shared(const int32_t *p) {
    int v;
    asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"(smem_addr(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_shared(int32_t *p, int v) {
    asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"(smem_addr(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int vload(const int32_t *p) { return *reinterpret_cast<const volatile int32_t *>(p); }
__device__ __forceinline__ void vstore(int32_t *p, int v) { *reinterpret_cast<volatile int32_t *>(p) = v; }
// generic address: a shared ring slot or a global face entry
__device__ __forceinline__ void st_entry(unsigned long long *p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.u64 [%0], %1;" ::"l"(p), "l"(v));
}
__device__ __forceinline__ unsigned long long ld_global_relaxed(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ ulonglong2 ld_global_relaxed_v2(const unsigned long long *p) {
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
    return v;
}

// Mark the column failed (first failure wins the launch status).
__device__ void c3_fail(C3Smem &sm, const LaunchDesc &L) {
    vstore(&sm.failed, 1);
    atomicCAS(L.err, 0, MSA_ETIMEOUT);
}

// The ring entries of a chunk of CH consecutive CTA times.
constexpr int CH = c3::CH;
struct C3Chunk {
    unsigned long long e[CH];
};
__device__ __forceinline__ C3Chunk c3_ring_load(const unsigned long long *p) {
    C3Chunk k;
#pragma unroll
    for (int j = 0; j < CH; ++j) k.e[j] = lds_u64_volatile(p + j * 32);
    return k;
}
__device__ __forceinline__ bool c3_ring_ready(const C3Chunk &k, int T) {  // this lane's entries carry T, T + 1, ..
    bool ok = true;
#pragma unroll
    for (int j = 0; j < CH; ++j) ok = ok && (int)(k.e[j] >> 32) == T + j;
    return ok;
}

// Slow path of a ring read: wait (bounded) until every lane's entries of the chunk carry their tags.
__device__ __noinline__ C3Chunk c3_ring_wait(const unsigned long long *p, int T, C3Smem &sm, const LaunchDesc &L) {
    C3Chunk k = c3_ring_load(p);
    uint64_t t0 = 0;
    for (int polls = 0; !__all_sync(kFull, c3_ring_ready(k, T)); ++polls) {
        if (polls >= 8) {
            if (t0 == 0) t0 = global_ns();
            if (vload(&sm.failed) || (int64_t)(global_ns() - t0) > L.spin_ns) {
                if ((threadIdx.x & 31) == 0) c3_fail(sm, L);
#pragma unroll
                for (int j = 0; j < CH; ++j) k.e[j] = pack_entry(kNeg, T + j);
                return k;
            }
            __nanosleep(20);
        }
        k = c3_ring_load(p);
    }
    return k;
}

// Registers of one compute lane that change from step to step.
struct C3St {
    int V[c3::R];       // V(T-1, r) on entry to step T, V(T, r) after it
    int P[c3::R];       // max over every candidate of cell (T, r) but e1
    int D[c3::R];       // max of the e02 and e012 candidates of cell (T+1, r)
    int pp[c3::R];      // p12 + 1 of the last R positions: shift register by position
    int S[c3::R];       // lane l-1's V(T-1, r), shuffled as soon as step T-1 had it
    int SM;             // lane l-1's V(T-1, -1)
    int f[c3::R];       // lane 0's inputs of step T (the staged face), loaded a step ahead
    int fm;
    C3Chunk cur, nxt;   // row -1 of this chunk's times and of the next chunk's
    int st_seen, dn_seen, fail_seen;  // the staged times, the warp below's progress and the column's failure,
                                      // read a step before their use
    int q;              // p02 entry of the next block on its way into the ring
};

// Constants of one compute lane for a column.
struct C3Ln {
    int p01[c3::R];     // pair score (x0, x1) + 4 per row
    int wR;             // first CTA row of the warp
    int tagout;         // tag base of ring-out entries (0: shared ring, epoch << 16: global face)
    int tagf1;          // tag base of this column's F1 entries
    bool last;          // lane 31's values are the F1 face
    int *f1b;           // f1b[w]
    int f1t;            // the step (of HF) of the F1 entry this lane writes
    int ctime;          // CTA time at which this lane computes the far corner (else never)
    int crow;           // the corner's row among this lane's R rows
    int N;              // CTA times of the column
    const int32_t *prog_dn;  // progress of the warp below (the last warp: its own)
    int wcorner;        // W of the far corner: the recorded key is V + W
    int32_t *qcorner;   // where the corner's key goes (for the traceback's cross-check)
};

// Addresses of the block of U steps starting at CTA time T0.
struct C3Blk {
    const unsigned long long *rin;  // ring[w][T0 mod SI][lane]
    const unsigned long long *rin2; // ring[w][(T0 + U) mod SI][lane]
    unsigned long long *rout;       // ring[w+1][T0 mod SI][lane] or F0[T0][lane] (generic)
    const int *f1row;               // f1r[T0 mod SF]
    unsigned char *tbp;             // traceback bytes of (T0, w, lane): R bytes
    unsigned long long *f1o;        // this lane's entry of F1[T0 ..][wR ..]
    const int *p02;                 // p02r[w][0][(T0 + 2 - wR - lane) mod SQ]
    const int *p12;                 // p12r[(T0 + 2 - wR) mod SP][lane]
    int *kept;                      // kept scores of (T0, w, lane): R / 4 runs of 4 words (kernels that keep them)
};

// Every HF steps a warp handles HF x R = 32 entries, one a lane: of face F1, and of
// its p02 ring, which is filled a block ahead: for the HF steps starting at CTA time
// T0 this lane's entry is row lane mod R at tau = T0 + 2 - wR + lane / R.
constexpr int HF = 32 / c3::R;
struct C3Fill {
    const uint16_t *c2;   // c2off entry of this lane's tau at T0 = 0
    const int *row;       // table row of the code of this lane's row
    int tau;              // this lane's tau at T0 = 0
    int *ring;            // p02r[w] of this lane's row
};
__device__ __forceinline__ void c3_fill_store(const C3Fill &f, int T0, int v) {
    const int slot = (f.tau + T0) & (c3::SQ - 1);
    f.ring[slot * 4] = v;
    f.ring[(slot < c3::U ? slot + c3::SQ : slot) * 4] = v;  // no branch: the step stays one basic block
}
__device__ __forceinline__ int c3_fill_load(const C3Fill &f, int T0) { return f.row[f.c2[T0]] - 5; }

// Lane 0's inputs of the step with staged-face row fr.
__device__ __forceinline__ void c3_load_face(C3St &g, const int *fr, int wR) {
#pragma unroll
    for (int r = 0; r < c3::R; r += 4) {
        const int4 v = *reinterpret_cast<const int4 *>(fr + 4 + wR + r);
        g.f[r] = v.x, g.f[r + 1] = v.y, g.f[r + 2] = v.z, g.f[r + 3] = v.w;
    }
    g.fm = fr[3 + wR];
}

// One step. Everything with a latency is started a step or more before its use:
// the shuffles of this step's values (for the next step) as soon as they exist,
// the staged face a step ahead, row -1 a chunk ahead with one vote per chunk.
template <int s, bool CAP, bool KEEP>
__device__ __forceinline__ void c3_step(C3St &g, const C3Ln &c, const C3Fill &f, const C3Blk &b, int T0, int lane,
                                        C3Smem &sm, const LaunchDesc &L) {
    constexpr int R = c3::R, H = c3::U, M = R - 1;
    static_assert(R == 4 || R == 8, "rows per warp: 4 or 8");
    static_assert(H % CH == 0 && H % R == 0 && H % HF == 0, "a block is a whole number of pair-score shifts");
    const int T = T0 + s;
    // p12 of the position x2 = T + 2 - lane - wR (row 0 of time T + 2), p02 of every row of time T + 2
    const int ppR = g.pp[s & M];  // position s - R, the last row's e12 pair
    g.pp[s & M] = b.p12[s * 32];
    int p02[R];
#pragma unroll
    for (int r = 0; r < R; r += 4) {
        const int4 v = *reinterpret_cast<const int4 *>(b.p02 + r * (c3::SQ + c3::U) + s * 4);
        p02[r] = v.x, p02[r + 1] = v.y, p02[r + 2] = v.z, p02[r + 3] = v.w;
    }
    // row -1 of the next chunk
    if constexpr (s % CH == 0)
        g.nxt = c3_ring_load(s + CH < H ? b.rin + (s + CH) * 32 : b.rin2 + (s + CH - H) * 32);
    // U(T, r) from lane l-1 (lane 0: the staged face)
    int Un[R];
#pragma unroll
    for (int r = 0; r < R; ++r) Un[r] = lane == 0 ? g.f[r] : g.S[r];
    const int UMn = lane == 0 ? g.fm : g.SM;
    const int VMn = (int)(unsigned)g.cur.e[s % CH];
    // the cells of time T: best candidate and its tag; the tags are the traceback bytes
    int acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        acc[r] = __viaddmax_s32(Un[r], 5, g.P[r]);
        g.V[r] = acc[r] & ~7;
        g.S[r] = __shfl_up_sync(kFull, g.V[r], 1);
    }
    g.SM = __shfl_up_sync(kFull, VMn, 1);
    if constexpr (CAP) {  // one lane of the launch, once
        if (T == c.ctime) {
#pragma unroll
            for (int r = 0; r < R; r += 4)
                *reinterpret_cast<int4 *>(sm.corner + r) = make_int4(g.V[r], g.V[r + 1], g.V[r + 2], g.V[r + 3]);
        }
    }
    // outputs: last row to the warp below (or face F0), traceback bytes, lane 31 to face F1
    st_entry(b.rout + s * 32, pack_entry(g.V[R - 1], c.tagout + T));
    c3_load_face(g, b.f1row + (s + 1) * c3::F1S, c.wR);
    unsigned pk[R / 4];
#pragma unroll
    for (int r = 0; r < R; r += 4)
        pk[r / 4] = __byte_perm(__byte_perm((unsigned)acc[r], (unsigned)acc[r + 1], 0x0040),
                                __byte_perm((unsigned)acc[r + 2], (unsigned)acc[r + 3], 0x0040), 0x5410) &
                    0x07070707u;
    if constexpr (R == 4)
        *reinterpret_cast<uint32_t *>(b.tbp + s * (c3::W * 32 * R)) = pk[0];
    else
        *reinterpret_cast<uint2 *>(b.tbp + s * (c3::W * 32 * R)) = make_uint2(pk[0], pk[R / 4 - 1]);
    if constexpr (KEEP) {
#pragma unroll
        for (int r = 0; r < R; r += 4)
            *reinterpret_cast<int4 *>(b.kept + s * (c3::W * 32 * R) + r * 32) = make_int4(acc[r], acc[r + 1], acc[r + 2], acc[r + 3]);
    }
    // a p02 entry of the next block: looked up in the first of HF steps, stored in the last
    if constexpr (s % HF == 0) g.q = c3_fill_load(f, T + H);
    if constexpr (s % HF == HF - 1) c3_fill_store(f, T - HF + 1 + H, g.q);
    // lane 31's values are the warp's part of face F1: laid out in shared memory and,
    // every HF steps, written by the whole warp, an entry per lane
    if (c.last) {
#pragma unroll
        for (int r = 0; r < R; r += 4)
            *reinterpret_cast<int4 *>(c.f1b + s % (2 * HF) * R + r) = make_int4(g.V[r], g.V[r + 1], g.V[r + 2], g.V[r + 3]);
    }
    int fo = 0;
    if constexpr (s % HF == HF - 1) {
        __syncwarp();
        fo = c.f1b[s / HF % 2 * 32 + lane];
    }
    if constexpr (s == H - 1) {
        g.st_seen = ld_acquire_shared(&sm.staged);
        g.dn_seen = ld_acquire_shared(c.prog_dn);
        g.fail_seen = vload(&sm.failed);
    }
    // P of time T + 1 and D of time T + 2
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int vm = (r ? g.V[r - 1] : VMn) + 7;
        const int y = (r ? Un[r - 1] : UMn) + c.p01[r];
        int pn = __viaddmax_s32(g.V[r], 3, y);
        pn = __viaddmax_s32(Un[r], r + 1 < R ? g.pp[(s - r - 1) & M] : ppR, pn);
        g.P[r] = __vimax3_s32(pn, g.D[r], vm);
        g.D[r] = __viaddmax_s32(y, g.pp[(s - r) & M], vm) + p02[r];
    }
    if constexpr (s % HF == HF - 1) st_entry(b.f1o + (s - HF + 1) * c3::WR, pack_entry(fo, c.tagf1 + T - HF + 1 + c.f1t));
    if constexpr (s % CH == CH - 1) {
        if (s + 1 < H || T + 1 < c.N) {  // no entry follows the column's last time
            if (__any_sync(kFull, !c3_ring_ready(g.nxt, T + 1)))
                g.nxt = c3_ring_wait(s + 1 < H ? b.rin + (s + 1) * 32 : b.rin2, T + 1, sm, L);
        }
        g.cur = g.nxt;
    }
}

// The unrolled steps of a block.
template <bool CAP, bool KEEP, int... S>
__device__ __forceinline__ void c3_steps(C3St &g, const C3Ln &c, const C3Fill &f, const C3Blk &b, int T0, int lane,
                                         C3Smem &sm, const LaunchDesc &L, std::integer_sequence<int, S...>) {
    (c3_step<S, CAP, KEEP>(g, c, f, b, T0, lane, sm, L), ...);
}

struct C3Col {
    int A, B, N;
    const unsigned long long *f0up, *f1left, *f1diag;  // producer faces (nullptr: none)
    unsigned long long *f0dst, *f1dst;                  // this column's faces
    int tagbase;                                        // (epoch << 16) of this launch
    const int *row1;                                    // table row of the code of x1 = 32B + lane
    const uint16_t *c2;                                 // c2off entry of x2 = -lane
};

// Staging warps: they copy the column's inputs from the producer columns' faces as
// soon as the entries' tags show this launch's values. Positions a producer never
// computes (past its last step, or no producer at all) are staged as kNeg.
//
// Waits of the staging warps, every sixteenth poll: true when the column failed or the limit ran out.
__device__ __forceinline__ bool c3_stage_expired(C3Smem &sm, uint64_t &t0, int lane, const LaunchDesc &L) {
    if (t0 == 0) t0 = global_ns();
    const bool end = vload(&sm.failed) || ld_volatile(L.err) != 0 || (int64_t)(global_ns() - t0) > L.spin_ns;
    if (!__any_sync(kFull, end)) return false;
    if (lane == 0 && !vload(&sm.failed)) c3_fail(sm, L);
    return true;
}
// Bounded wait until the first n of prog have reached need.
__device__ __forceinline__ bool c3_wait_room(C3Smem &sm, const int32_t *prog, int n, int need, int lane,
                                             const LaunchDesc &L) {
    uint64_t t0 = 0;
    for (int polls = 0; !__all_sync(kFull, lane >= n || ld_acquire_shared(prog + lane) >= need); ++polls) {
        if ((polls & 15) == 15 && c3_stage_expired(sm, t0, lane, L)) return false;
        __nanosleep(100);
    }
    return true;
}

// Row warp: face F0 of the column above into ring[0], SB CTA times a batch. The
// ring's entries carry their own tags, so a lane stores what it has.
__device__ void c3_stage_rows(C3Smem &sm, const C3Col &cc, int lane, const LaunchDesc &L) {
    constexpr int SB = c3::SB, NL = SB / 2;                // loads per lane and batch (2 rows per load)
    const int half = lane >> 4, pair = 2 * (lane & 15);    // row parity, first entry
    const ulonglong2 none = make_ulonglong2(pack_entry(kNeg, 0), pack_entry(kNeg, 0));
    ulonglong2 e[NL];
    int room = -c3::U + c3::SI;  // ring slots of the CTA times below are free
    for (int Ts = -c3::U; Ts < cc.N; Ts += SB) {
        // the slots to fill must have been read by warp 0
        if (room < Ts + SB && !c3_wait_room(sm, &sm.prog[0], 1, Ts + SB - c3::SI, lane, L)) return;
        room = ld_acquire_shared(&sm.prog[0]) + c3::SI;
        uint64_t t0 = 0;
        for (int polls = 0;; ++polls) {
            bool ok = true;
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int T = Ts + 2 * i + half;
                e[i] = none;
                if (cc.f0up && T + c3::WR < cc.N)
                    e[i] = ld_global_relaxed_v2(cc.f0up + (int64_t)(T + c3::WR + c3::U) * 32 + pair);
            }
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int T = Ts + 2 * i + half, want = cc.tagbase + T + c3::WR;
                if (cc.f0up && T + c3::WR < cc.N)
                    ok = ok && (int)(e[i].x >> 32) == want && (int)(e[i].y >> 32) == want;
            }
            if (__all_sync(kFull, ok)) break;
            if ((polls & 15) == 15 && c3_stage_expired(sm, t0, lane, L)) return;
        }
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            const int T = Ts + 2 * i + half;
            *reinterpret_cast<ulonglong2 *>(&sm.ring[0][T & (c3::SI - 1)][pair]) =
                make_ulonglong2(pack_entry((int)(unsigned)e[i].x, T), pack_entry((int)(unsigned)e[i].y, T));
        }
    }
}

// Column warp: face F1 of the column to the left and the corner of the column
// above-left into f1r, and the (axis 1, axis 2) pair scores into p12r; it
// publishes how many CTA times are staged.
__device__ void c3_stage_cols(C3Smem &sm, const C3Col &cc, int lane, const LaunchDesc &L) {
    constexpr int SB = 8;                                          // CTA times per batch: 0.642 ms, 4: 0.69
    constexpr int LPR = c3::WR / 2, RPL = 32 / LPR, NL = SB / RPL;  // lanes per row, rows per load, loads
    static_assert(SB % RPL == 0 && 32 % LPR == 0, "F1 rows per load");
    const int sub = lane / LPR, pair = 2 * (lane % LPR);
    const ulonglong2 none = make_ulonglong2(pack_entry(kNeg, 0), pack_entry(kNeg, 0));
    for (int Ts = -c3::U; Ts < cc.N; Ts += SB) {
        // the slots to fill must have been read by every compute warp
        if (!c3_wait_room(sm, sm.prog, c3::W, Ts + SB - c3::SF, lane, L)) return;
        ulonglong2 e[NL];
        unsigned long long d;  // lane i: the corner of the batch's row i
        uint64_t t0 = 0;
        for (int polls = 0;; ++polls) {
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int T = Ts + RPL * i + sub;
                e[i] = none;
                if (cc.f1left && T + 31 < cc.N)
                    e[i] = ld_global_relaxed_v2(cc.f1left + (int64_t)(T + 31 + c3::U) * c3::WR + pair);
            }
            const int Td = Ts + lane;
            d = pack_entry(kNeg, 0);
            const bool corner = lane < SB && cc.f1diag && Td + 31 + c3::WR < cc.N;
            if (corner) d = ld_global_relaxed(cc.f1diag + (int64_t)(Td + 31 + c3::WR + c3::U) * c3::WR + c3::WR - 1);
            if (polls == 0) {
                // p12 of the batch's rows (warp 0 reads row T + 2 at time T), while the loads fly
#pragma unroll
                for (int i = 0; i < SB; ++i) {
                    const int t = Ts + i + 2;
                    const int slot = t & (c3::SP - 1), v = cc.row1[cc.c2[t]] + 1;
                    sm.p12r[slot][lane] = v;
                    if (slot < c3::U) sm.p12r[slot + c3::SP][lane] = v;
                }
            }
            bool ok = !corner || (int)(d >> 32) == cc.tagbase + Td + 31 + c3::WR;
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int T = Ts + RPL * i + sub, want = cc.tagbase + T + 31;
                if (cc.f1left && T + 31 < cc.N)
                    ok = ok && (int)(e[i].x >> 32) == want && (int)(e[i].y >> 32) == want;
            }
            if (__all_sync(kFull, ok)) break;
            if ((polls & 15) == 15 && c3_stage_expired(sm, t0, lane, L)) return;
        }
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            const int T = Ts + RPL * i + sub;
            *reinterpret_cast<int2 *>(&sm.f1r[T & (c3::SF - 1)][4 + pair]) =
                make_int2((int)(unsigned)e[i].x, (int)(unsigned)e[i].y);
        }
        if (lane < SB) sm.f1r[(Ts + lane) & (c3::SF - 1)][3] = (int)(unsigned)d;
        __syncwarp();
        if (lane == 0) st_release_shared(&sm.staged, Ts + SB);
    }
}

// Block prologue of a compute warp: publish progress, then wait (bounded) until
// the staged face covers the block and the warp below has freed the ring slots.
// The values seen are loads of the previous block's end.
__device__ __forceinline__ bool c3_block_wait(C3Smem &sm, const C3Ln &c, int w, int T0, const C3St &g,
                                              const LaunchDesc &L) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) st_release_shared(&sm.prog[w], T0);
    const int need_st = T0 + c3::U;
    const int need_dn = w == c3::W - 1 ? -(1 << 30) : T0 + c3::U - c3::SI;
    if (__all_sync(kFull, g.st_seen >= need_st && g.dn_seen >= need_dn && !g.fail_seen)) return true;
    uint64_t t0 = 0;
    for (int polls = 0;; ++polls) {
        if (!__any_sync(kFull, vload(&sm.failed) != 0) &&
            __all_sync(kFull, ld_acquire_shared(&sm.staged) >= need_st && ld_acquire_shared(c.prog_dn) >= need_dn))
            return true;
        if (__any_sync(kFull, vload(&sm.failed) != 0)) return false;
        if (polls < 4) continue;
        if (t0 == 0) t0 = global_ns();
        if (__any_sync(kFull, (int64_t)(global_ns() - t0) > L.spin_ns)) {
            if ((threadIdx.x & 31) == 0) c3_fail(sm, L);
            return false;
        }
        __nanosleep(32);
    }
}

}  // namespace

// CAP: the lane that computes the far corner lays its rows out in shared memory at the
// corner's CTA time and records the corner's key at the column's end, for the
// traceback's cross-check: a comparison and two predicated stores per step, 0.703 ms at
// 700 x 760 x 800 and 0.107 at 128^3 (plain launches, without it, 0.640 and 0.099). A
// second copy of the block's steps with the capture, for the corner's block only, was
// 1.96 and 0.232 (instruction fetch). KEEP: every cell's
// best candidate, V plus tag, is kept for the near-optimal walk (c3::kept_term): the
// traceback's layout with a word for its byte and a lane's rows in runs of four, so
// that each 16-byte store of a warp is one run (120 x 110 x 130: 0.089 ms, 0.085 without
// KEEP); the corner's lane reads its own store back.
template <bool CAP, bool KEEP>
__global__ void __launch_bounds__(c3::THREADS, c3::CTAS) fill_col3_kernel(const LaunchDesc L) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C3Smem &sm = *reinterpret_cast<C3Smem *>(smem_raw);
    int *tabr = reinterpret_cast<int *>(smem_raw + sizeof(C3Smem));
    uint16_t *c2off = reinterpret_cast<uint16_t *>(tabr + L.tab_ints);  // axis-2 codes by x2 + CODEPAD

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid == 0) sm.cur_prob = -1;
    __syncthreads();

    while (true) {
        if (tid == 0) {
            sm.ctl[0] = atomicAdd(L.ticket, 1);
            sm.ctl[1] = ld_volatile(L.err);
        }
        __syncthreads();
        const int ticket = sm.ctl[0];
        const int errnow = sm.ctl[1];
        __syncthreads();
        if ((int64_t)ticket >= L.ntickets || errnow != 0) break;

        const uint64_t ent = L.order[ticket];
        const int pidx = (int)(ent >> 32);
        const ProblemDesc &P = L.probs[pidx];
        if (ld_volatile(&P.istat->status) != 0) continue;  // uniform: every thread reads the same word
        const int lin = (int)(uint32_t)ent;
        const int NB = P.G[1];
        C3Col cc;
        cc.A = lin / NB;
        cc.B = lin - cc.A * NB;
        cc.N = c3::nsteps(P.rho[2]);
        const int64_t f0s = P.face0_stride / 2, f1s = P.face1_stride / 2;  // entries per column face
        unsigned long long *F0 = reinterpret_cast<unsigned long long *>(P.Q);
        unsigned long long *F1 = reinterpret_cast<unsigned long long *>(P.aux);
        cc.f0dst = F0 + (int64_t)lin * f0s;
        cc.f1dst = F1 + (int64_t)lin * f1s;
        cc.f0up = cc.A > 0 ? F0 + (int64_t)(lin - NB) * f0s : nullptr;
        cc.f1left = cc.B > 0 ? F1 + (int64_t)(lin - 1) * f1s : nullptr;
        cc.f1diag = (cc.A > 0 && cc.B > 0) ? F1 + (int64_t)(lin - NB - 1) * f1s : nullptr;
        cc.tagbase = L.epoch << 16;
        // a withheld column (test hook) writes faces no reader accepts
        const int tag_faces = (int64_t)ticket == L.withhold ? 0 : cc.tagbase;

        const int A = P.A;
        // pair table with a sentinel code A for positions x2 <= 0, and the axis-2 codes
        const int have = sm.cur_prob;
        __syncthreads();
        if (have != pidx)
            for (int i = tid; i < A * (A + 1); i += c3::THREADS) {
                const int c0 = i / (A + 1), c2 = i % (A + 1);
                tabr[i] = c2 == A ? c3::kSentinelPair : P.tab[c0 * A + c2];
            }
        if (tid == 0) {
            sm.cur_prob = pidx;
            sm.staged = -c3::U;
            sm.failed = 0;
        }
        if (tid < c3::W) sm.prog[tid] = -c3::U;
        const int len2 = P.len[2];
        for (int i = tid; i < P.rho[2] + 2 * c3::CODEPAD + 16; i += c3::THREADS) {
            const int x2 = i - c3::CODEPAD;  // position x2 consumes residue x2 - 1
            c2off[i] = (uint16_t)(x2 <= 0 ? A : x2 <= len2 ? P.codes[P.cofs[2] + x2 - 1] : 0);
        }
        // pair scores before the first block belong to positions x2 < 0
        for (int i = tid; i < (c3::SP + c3::U) * 32; i += c3::THREADS) (&sm.p12r[0][0])[i] = c3::kSentinelPair;
        for (int i = tid; i < c3::W * (c3::SQ + c3::U) * c3::R; i += c3::THREADS)
            (&sm.p02r[0][0][0][0])[i] = c3::kSentinelPair;
        // ring entries start with a tag no step uses
        for (int i = tid; i < c3::W * c3::SI * 32; i += c3::THREADS)
            (&sm.ring[0][0][0])[i] = pack_entry(kNeg, 0x7fffffff);
        __syncthreads();

        const int x1 = cc.B * 32 + lane;
        const int code1 = (x1 >= 1 && x1 <= P.len[1]) ? P.codes[P.cofs[1] + x1 - 1] : 0;
        if (w == c3::W) {
            c3_stage_rows(sm, cc, lane, L);
        } else if (w > c3::W) {
            cc.row1 = tabr + code1 * (A + 1);
            cc.c2 = c2off + c3::CODEPAD - lane;
            c3_stage_cols(sm, cc, lane, L);
        } else {
            const bool lastw = w == c3::W - 1;
            C3Ln c;
            c.wR = w * c3::R;
            c.last = lane == 31;
            c.f1b = &sm.f1b[w][0][0];
            c.f1t = lane / c3::R;
            c.tagout = lastw ? tag_faces : 0;
            c.tagf1 = tag_faces;
            c.N = cc.N;
            c.prog_dn = &sm.prog[lastw ? w : w + 1];
            const int x0b = cc.A * c3::WR + c.wR;
            auto code0 = [&](int r) {
                const int x0 = x0b + r;
                return (x0 >= 1 && x0 <= P.len[0]) ? (int)P.codes[P.cofs[0] + x0 - 1] : 0;
            };
#pragma unroll
            for (int r = 0; r < c3::R; ++r) c.p01[r] = P.tab[code0(r) * A + code1] + 4;
            C3Fill f;
            f.row = tabr + code0(lane % c3::R) * (A + 1);
            f.tau = 2 - c.wR + lane / c3::R;
            f.c2 = c2off + c3::CODEPAD + f.tau - lane % c3::R;
            f.ring = &sm.p02r[w][lane % c3::R / 4][0][lane % 4];
#pragma unroll
            for (int n = -c3::U; n < 0; n += HF) c3_fill_store(f, n, c3_fill_load(f, n));
            {  // the far corner (len0, len1, len2): row rho of lane l at CTA time len2 + l + rho
                const int rhoc = P.len[0] - cc.A * c3::WR, lc = P.len[1] - 32 * cc.B;
                const bool mine = rhoc >= c.wR && rhoc < c.wR + c3::R && lc == lane;
                c.ctime = mine ? P.len[2] + lc + rhoc : (int)0x80000000;
                c.crow = rhoc - c.wR;
                c.wcorner = P.w_corner;
                c.qcorner = P.qcorner;
            }

            C3St g;
#pragma unroll
            for (int r = 0; r < c3::R; ++r) {
                g.V[r] = kNeg;
                g.P[r] = kNeg;
                g.D[r] = kNeg;
                g.S[r] = kNeg;
            }
            const bool origin = cc.A == 0 && cc.B == 0 && w == 0 && lane == 0;
            g.SM = kNeg;
            g.st_seen = g.dn_seen = -(1 << 30);
            g.fail_seen = 0;
            g.cur = c3_ring_wait(&sm.ring[w][-c3::U & (c3::SI - 1)][lane], -c3::U, sm, L);
            // p12 of the positions before time -U, all below 0
#pragma unroll
            for (int j = 0; j < c3::R; ++j) g.pp[j] = c3::kSentinelPair;

            unsigned long long *ringout = lastw ? cc.f0dst + lane : &sm.ring[w + 1][0][lane];
            unsigned char *tbw = P.tb + (int64_t)lin * c3::tb_col_bytes(P.rho[2]) + (w * 32 + lane) * c3::R;
            C3Blk b;
            b.rin2 = &sm.ring[w][-c3::U & (c3::SI - 1)][lane];
            b.rout = ringout + (lastw ? 0 : (-c3::U & (c3::SI - 1)) * 32);
            b.f1row = &sm.f1r[-c3::U & (c3::SF - 1)][0];
            b.tbp = tbw;
            b.kept = KEEP ? P.kept + (int64_t)lin * c3::tb_col_bytes(P.rho[2]) + w * (32 * c3::R) + lane * 4 : nullptr;
            b.f1o = cc.f1dst + (int64_t)c.f1t * c3::WR + c.wR + lane % c3::R;
            b.p02 = &sm.p02r[w][0][(-c3::U + 2 - c.wR - lane) & (c3::SQ - 1)][0];
            b.p12 = &sm.p12r[(-c3::U + 2 - c.wR) & (c3::SP - 1)][lane];
            for (int T0 = -c3::U; T0 < cc.N; T0 += c3::U) {
                if (!c3_block_wait(sm, c, w, T0, g, L)) break;
                if (T0 == 0 && origin) g.P[0] = 0;  // H(0) = 0, no move
                c3_load_face(g, b.f1row, c.wR);
                b.rin = b.rin2;
                b.rin2 = &sm.ring[w][(T0 + c3::U) & (c3::SI - 1)][lane];
                // the next block's addresses, formed while this one runs
                C3Blk n;
                const int Tn = T0 + c3::U;
                n.rin2 = b.rin2;
                n.rout = lastw ? b.rout + c3::U * 32 : ringout + (Tn & (c3::SI - 1)) * 32;
                n.f1row = &sm.f1r[Tn & (c3::SF - 1)][0];
                n.tbp = b.tbp + c3::U * (c3::W * 32 * c3::R);
                n.kept = KEEP ? b.kept + c3::U * (c3::W * 32 * c3::R) : nullptr;
                n.f1o = b.f1o + c3::U * c3::WR;
                n.p02 = &sm.p02r[w][0][(Tn + 2 - c.wR - lane) & (c3::SQ - 1)][0];
                n.p12 = &sm.p12r[(Tn + 2 - c.wR) & (c3::SP - 1)][lane];
                c3_steps<CAP, KEEP>(g, c, f, b, T0, lane, sm, L, std::make_integer_sequence<int, c3::U>{});
                b = n;
            }
            if (CAP && c.ctime != (int)0x80000000) __stcg(c.qcorner, sm.corner[c.crow] + c.wcorner);
            if constexpr (KEEP) {  // the corner's lane has its score from its own store
                if (c.ctime != (int)0x80000000) {
                    const int64_t at = c3::kept_term(0, P.len[0], NB, P.rho[2]) + c3::kept_term(1, P.len[1], NB, P.rho[2]) +
                                       c3::kept_term(2, P.len[2], NB, P.rho[2]);
                    __stcg(c.qcorner, (*reinterpret_cast<volatile int *>(P.kept + at) & ~7) + c.wcorner);
                }
            }
            __syncwarp();
            if (lane == 0) st_release_shared(&sm.prog[w], 1 << 30);
        }
        __syncthreads();
        if (vload(&sm.failed)) break;
    }
}

// Dynamic shared memory: rings and staged faces, the pair table with its sentinel
// column (A*(A+1) entries) and the axis-2 codes.
int col3_smem_bytes(int alphabet_size) {
    return (int)sizeof(C3Smem) + alphabet_size * (alphabet_size + 1) * 4 +
           (c3::MAXRHO2 + 2 * c3::CODEPAD + 16) * 2 + 16;
}

// The attribute allows the largest alphabet's layout; set once per device.
cudaError_t col3_attributes() {
    static DeviceOnce once;
    return once.run([] {
        cudaError_t e = cudaSuccess;
        for (auto kernel : {fill_col3_kernel<false, false>, fill_col3_kernel<true, false>, fill_col3_kernel<false, true>})
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, col3_smem_bytes(c3::MAXA));
        return e;
    });
}

int fill_col3_ctas_per_sm(int smem) {
    if (col3_attributes() != cudaSuccess) return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fill_col3_kernel<false, false>, c3::THREADS, smem) != cudaSuccess)
        return 0;
    return n;
}

cudaError_t launch_fill_col3(const LaunchDesc &L, int grid, int smem, cudaStream_t s) {
    cudaError_t e = col3_attributes();
    if (e != cudaSuccess) return e;
    if (smem > col3_smem_bytes(c3::MAXA)) return cudaErrorInvalidValue;
    if (L.keep)
        fill_col3_kernel<false, true><<<grid, c3::THREADS, smem, s>>>(L);
    else if (L.corner)
        fill_col3_kernel<true, false><<<grid, c3::THREADS, smem, s>>>(L);
    else
        fill_col3_kernel<false, false><<<grid, c3::THREADS, smem, s>>>(L);
    return cudaGetLastError();
}

}  // namespace msadp
