// Streamed line fill for k = 4..6: the line kernel's recurrence and lanes
// (fill_lines.cuh: lane l of a warp owns one line of a 32-line block, skewed by
// the sum of its local coordinates; the moves that also advance the last axis s are
// folded from the previous position's candidates), organised for the latency of the
// hardware. Measured (fill), with the exchange on warps of its own against inside the
// sweep: k5 protein 33 - 45 1.097 against 1.402 ms, 15^5 0.100 / 0.159, 31^5 0.407 / 0.594;
// k4 DNA 110 - 130 0.898 / 0.946, 61 - 64 0.184 / 0.237, 41^4 0.103 / 0.147, 21^4 0.050 /
// 0.066.
//
// * A CTA of W sweeping warps owns a SUPER-BLOCK of W line blocks (a grid of extents
//   stream_wg over the line axes) and sweeps it over the WHOLE last axis in
//   lockstep: at step t every lane of the sweep computes position z = t - sigma of
//   its line, sigma being the sum of the line's coordinates inside the
//   super-block, and a barrier of the sweep's warps ends the step. Every predecessor
//   line of the super-block then holds position z at time t - |m'|, so warps exchange
//   nothing but shared memory; only super-blocks talk through global memory.
//   The skew, the set-up and the ticket are paid once per super-block column.
// * Super-blocks are handed out in wave order of their grid (section 3: blocks
//   whose coordinates sum to w form wave w). What a super-block's upper-face lines held
//   at the U TIMES of a block goes out as (value, tag) 8-byte entries (the tag is the
//   launch's epoch). Publishing by time makes a block's data complete as soon as the
//   block ends; a consumer's halo time tau is its producer's time tau + SB_S (the
//   super-block extents along the axes S in which the producer lies below).
// * Separate warps of the CTA do that exchange: they write the swept blocks' faces and
//   bring the halo of the blocks to come, loading entries until all carry the epoch (a
//   bounded wait), while the sweep runs; the sweep only looks, two steps before a block
//   ends, whether the next block's halo is there. In the sweeping warps themselves
//   (copies into a staging buffer during a block, tag checks and ring stores at its
//   end) the exchange took 106 of a step's 181 instructions at k = 5 and stood between
//   the blocks. Correctness rests on the tags, so no fence or release/acquire pair is
//   needed between CTAs: an aligned 8-byte entry is written by one store and read
//   whole, each entry is written once per launch, and earlier launches left smaller
//   epochs (the plan clears the faces before the first launch and when epochs wrap).
//
// Shared memory per CTA:
//   V      a ring of three blocks' times per line of the halo'd super-block (local
//          coordinates -1 .. SB_i - 1), indexed by time: position z of line c sits
//          in slot (z + sigma(c)) mod 3U. At step t every lane reads its predecessor
//          line c - e_m' at time t - |m'| and writes its own line's slot of time t: a
//          constant offset from the block's slots or from those of the block before, so
//          the steps are unrolled once. The 32 accesses of a warp are conflict-free when
//          sum_i c_i A_i is distinct mod 32 over a line block (strides A_i found by
//          exhaustive search, below). The third block's slots take the arriving halo.
//   PT     an R-position ring of the pair tables of s against every line axis, refilled
//          by the exchanging warps.
//   tables of the halo and face lines, the neighbour super-block of every
//          subset of the line axes, the residue code of every pair-table row.
//
// Global memory: the traceback bytes of each line block (a tile of the line
// kernel's layout 3 spanning the whole last axis: cell (c, z) at
// (z + sum c_i) * 32 + lane); the faces of each super-block: its upper-face
// lines, line-major, ZQ times each.
#pragma once

#include <type_traits>

#include "device_common.cuh"

namespace msadp {

// Ring slots per line: the block being swept, the one before and the one whose halo arrives.
__host__ __device__ constexpr int stream_ring_d(int K) { return 3 * stream_block(K); }
// Pair-table ring positions: two blocks and the skew of a super-block at least.
__host__ __device__ constexpr int stream_pt_ring(int K) { return K == 4 ? 64 : 32; }

// Ring stride (words) of line axis i over the halo'd super-block: the smallest
// footprint with every line's D slots disjoint and sum_i c_i A_i distinct mod 32
// over a warp's line block.
__host__ __device__ constexpr int stream_stride(int K, int i) {
    constexpr int k4[] = {217, 24, 1086}, k5[] = {362, 1812, 121, 24}, k6[] = {24, 362, 121, 1812, 5456};
    return K == 4 ? k4[i] : K == 5 ? k5[i] : k6[i];
}
template <int K>
__host__ __device__ constexpr int stream_move_off(int m) {
    int s = 0;
    for (int i = 0; i < K - 1; ++i)
        if ((m >> i) & 1) s += stream_stride(K, i);
    return s;
}
template <int K>
__host__ __device__ constexpr int stream_halo_lines() {  // lines of the halo'd super-block with some index -1
    int all = 1;
    for (int i = 0; i < K - 1; ++i) all *= stream_sb(K, i) + 1;
    return all - 32 * stream_warps(K);
}
template <int K>
__host__ __device__ constexpr int stream_rows() {  // pair-table rows: one per (line axis, coordinate)
    int n = 0;
    for (int i = 0; i < K - 1; ++i) n += stream_sb(K, i);
    return n;
}
template <int K>
__host__ __device__ constexpr int stream_ring_words() {
    int s = stream_ring_d(K);
    for (int i = 0; i < K - 1; ++i) s += stream_sb(K, i) * stream_stride(K, i);
    return round_up(s, 4);
}
// Warps of a CTA that exchange the faces: half or all of the sweep's. k = 4 with 4 / 8: 20^4
// 0.0527 / 0.0494 ms, 40^4 0.112 / 0.106; k = 5 with 1 / 2 / 4 / 8: 2.31 / 1.38 / 1.10 / 1.23.
__host__ __device__ constexpr int stream_xwarps(int K) { return K == 4 ? 8 : 4; }
// Shared memory of a CTA, in 4-byte words (every part 16-byte aligned).
template <int K>
struct StreamLayout {
    static constexpr int NH = stream_halo_lines<K>();
    static constexpr int NFL = stream_face_lines(K);
    static constexpr int NROW = stream_rows<K>();
    // pair-table rows: an R-position ring stored twice (slots p mod R and
    // p mod R + R, so that a block's positions need no wrap), rows staggered by
    // (a line block's skew) + 1 banks
    static constexpr int ZS = 2 * stream_pt_ring(K) + line_skew_max(K) + 1;
    static constexpr int NT = 32 * stream_warps(K);
    static constexpr int V = 0;
    static constexpr int PT = V + stream_ring_words<K>();
    static constexpr int HSRC = PT + round_up(NROW * ZS, 4);  // per halo line: its producer's face line (-1: none)
    static constexpr int HTAB = HSRC + round_up(NH, 4);
    static constexpr int FTAB = HTAB + round_up(NH, 4);
    static constexpr int NB = FTAB + round_up(NFL, 4);
    static constexpr int CROW = NB + round_up(1 << (K - 1), 4);
    static constexpr int MISC = CROW + round_up(NROW, 4);  // ticket, progress, verdicts
    static constexpr int WORDS = MISC + 8 + round_up(stream_xwarps(K), 4);
};
template <int K>
__host__ __device__ constexpr int stream_smem_bytes() {
    return StreamLayout<K>::WORDS * 4;
}
template <int K>
__host__ __device__ constexpr int stream_threads() {
    return 32 * stream_warps(K);
}
// The streamed kernel's CTA: the sweep's warps and those that exchange the faces.
template <int K>
__host__ __device__ constexpr int stream_cta_threads() {
    return stream_threads<K>() + 32 * stream_xwarps(K);
}
// CTAs per SM: what shared memory allows (228 KB per SM, 1 KB reserved per CTA)
// and what leaves the sweep its registers (it keeps 2^(k-1) pair sums live). k = 4 with a
// third CTA (56 registers): 0.941 against 0.949 ms, but 40^4 0.126 against 0.112; k = 5 with
// a fourth (64): 1.063 against 1.099, but 20^5 0.184 against 0.171.
template <int K>
__host__ __device__ constexpr int stream_min_ctas() {
    const int c = (228 * 1024) / (stream_smem_bytes<K>() + 1024), cr = K == 4 ? 2 : 3;
    return c < cr ? c : cr;
}

// Lines of a super-block and of its halo, numbered in closed form so that all
// threads fill a CTA's tables (one thread counting them took 0.02 ms at k = 4, 0.09 at
// k = 6 and 0.2 at k = 8, more than the sweep of a small problem): coordinates of line j (axis 0 most significant);
// the number of a face line (some c_i = SB_i - 1) among the face lines, else -1; and
// for halo'd index j (digits h_i in [0, SB_i]) its number among the halo lines (some
// h_i = 0), else -1.
template <int K>
__device__ __forceinline__ void super_line(int j, int (&c)[K - 1]) {
#pragma unroll
    for (int i = K - 2; i >= 0; --i) {
        c[i] = j % stream_sb(K, i);
        j /= stream_sb(K, i);
    }
}
template <int K>
__device__ __forceinline__ int face_number(const int (&c)[K - 1]) {
    int j = 0, inner = 0;  // the line's index; lines before it with every coordinate below SB_i - 1
    bool prefix = true;    // ... coordinates so far
#pragma unroll
    for (int i = 0; i < K - 1; ++i) {
        j = j * stream_sb(K, i) + c[i];
        inner = inner * (stream_sb(K, i) - 1) + (prefix ? c[i] : 0);
        prefix = prefix && c[i] < stream_sb(K, i) - 1;
    }
    return prefix ? -1 : j - inner;
}
template <int K>
__device__ __forceinline__ int halo_number(int j, int (&h)[K - 1]) {
    int rem = j;
#pragma unroll
    for (int i = K - 2; i >= 0; --i) {
        h[i] = rem % (stream_sb(K, i) + 1);
        rem /= stream_sb(K, i) + 1;
    }
    int inner = 0;  // indices before j with every digit >= 1
    bool prefix = true;
#pragma unroll
    for (int i = 0; i < K - 1; ++i) {
        inner = inner * stream_sb(K, i) + (prefix && h[i] >= 1 ? h[i] - 1 : 0);
        prefix = prefix && h[i] >= 1;
    }
    return prefix ? -1 : j - inner;
}

__device__ __forceinline__ ulonglong2 ld_relaxed_v2(const unsigned long long *p) {
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ int ld_acquire_shared(const int32_t *p) {
    int v;
    asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_shared(int32_t *p, int v) {
    asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
// The barrier of the sweep's warps.
template <int N>
__device__ __forceinline__ void sweep_barrier() {
    asm volatile("bar.sync 1, %0;" ::"n"(N) : "memory");
}
// Bounded wait of a sweep warp for the exchanging warp (whose own waits are bounded and
// which then sets `failed`); the same in every lane.
static __device__ __noinline__ bool stream_wait(const int32_t *landed, int n, int need, volatile int32_t *failed, int64_t spin_ns) {
    uint64_t t0 = 0;
    for (int polls = 0;; ++polls) {
        if (__all_sync(kFull, ld_acquire_shared(landed + (threadIdx.x & 31) % n) >= need)) return true;
        if ((polls & 15) == 15) {
            if (t0 == 0) t0 = global_ns();
            if (__any_sync(kFull, *failed != 0 || (int64_t)(global_ns() - t0) > 2 * spin_ns + 1000000000)) {
                *failed = 1;
                return false;
            }
        }
        __nanosleep(32);
    }
}
__device__ __forceinline__ void st_relaxed_v2(unsigned long long *p, unsigned long long a, unsigned long long b) {
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ unsigned long long tagged(int value, int tag) {
    return (unsigned long long)(unsigned)value | ((unsigned long long)(unsigned)tag << 32);
}

template <int K>
__global__ void __launch_bounds__(stream_cta_threads<K>(), stream_min_ctas<K>()) fill_lines_stream_kernel(const LaunchDesc L) {
    constexpr int NA = K - 1;
    constexpr int M = (1 << NA) - 1;
    constexpr int NS = stream_threads<K>(), NT = stream_cta_threads<K>();  // threads of the sweep, of the CTA
    constexpr int NLINES = NS;
    constexpr int SMAX = stream_skew_max(K);
    constexpr int U = stream_block(K), R = stream_pt_ring(K);
    constexpr int MASKB = (1 << K) - 1;
    using LY = StreamLayout<K>;
    constexpr int NH = LY::NH, NFL = LY::NFL, NROW = LY::NROW, ZS = LY::ZS;
    constexpr int LQ = U / 2, LG = 32 / LQ;        // lanes per line (two entries each), lines per load of the warp
    constexpr int NX = stream_xwarps(K);
    constexpr int HB = K == 4 ? 3 : 8;            // loads in flight per lane of an exchanging warp
    constexpr int PQ = (NROW * U + 32 * NX - 1) / (32 * NX);  // pair-table entries per lane and chunk
    constexpr int NBATCH = (NH + NX * LG * HB - 1) / (NX * LG * HB);  // batches of a chunk per exchanging warp
    // The ring holds three blocks of a line's times: the one being swept, the one before
    // (read up to k - 1 times back) and the one whose halo is arriving. The pair-table
    // ring: while block c - 1 is swept, it reads positions from (c - 1) U + 1 - SMAX on, and
    // chunk c's positions cU + 1 .. (c + 1) U replace those R below.
    static_assert(stream_ring_d(K) == 3 * U && U >= NA && U % 2 == 0 && 32 % LQ == 0 && (R & (R - 1)) == 0 &&
                      2 * U + SMAX <= R && LY::PT < (1 << 14) && NFL < 128 && M < 32,
                  "geometry");

    extern __shared__ __align__(16) unsigned char smem_raw[];
    int32_t *sm = reinterpret_cast<int32_t *>(smem_raw);
    int32_t *V = sm + LY::V;
    int32_t *PT = sm + LY::PT;
    int32_t *hsrc = sm + LY::HSRC;
    // halo lines: ring base | producer face line << 14 | axes S at -1 << 21 |
    // (the sum of SB_i over S: the producer's time offset) << 26
    uint32_t *htab = reinterpret_cast<uint32_t *>(sm + LY::HTAB);
    uint32_t *ftab = reinterpret_cast<uint32_t *>(sm + LY::FTAB);  // face lines: ring base
    int32_t *nb = sm + LY::NB;
    int32_t *crow = sm + LY::CROW;
    // [0] ticket, [1] blocks swept, [2] the waiting path's verdict, [3] failed, [4] [5] verdicts on
    // the next block's chunk (by block parity), [8 ..] chunks of the halo in place, per exchanging warp
    volatile int32_t *misc = sm + LY::MISC;
    int32_t *const swept = sm + LY::MISC + 1, *const landed = sm + LY::MISC + 8;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // face lines of the super-block in line order; their numbers index the faces
    for (int j = tid; j < NLINES; j += NT) {
        int c[NA], base = 0;
        super_line<K>(j, c);
        const int f = face_number<K>(c);
#pragma unroll
        for (int i = 0; i < NA; ++i) base += (c[i] + 1) * stream_stride(K, i);
        if (f >= 0) ftab[f] = (uint32_t)base;
    }
    // halo lines
    for (int j = tid; j < LY::NH + NLINES; j += NT) {
        int h[NA], c[NA], base = 0;
        uint32_t S = 0, sbs = 0;
        const int n = halo_number<K>(j, h);
        if (n < 0) continue;
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            base += h[i] * stream_stride(K, i);
            c[i] = h[i] == 0 ? stream_sb(K, i) - 1 : h[i] - 1;  // the line in the super-block that produces it
            if (h[i] == 0) {
                S |= 1u << i;
                sbs += stream_sb(K, i);
            }
        }
        htab[n] = (uint32_t)base | (uint32_t)face_number<K>(c) << 14 | S << 21 | sbs << 26;
    }

    // this thread's line: warp coordinates in the warp grid, lane coordinates in
    // the line block; ring base and skew inside the super-block
    int cl[NA], cw[NA];
    int vbase = 0, sig = 0, sigw = 0;
    {
        int rw = warp;
#pragma unroll
        for (int i = NA - 1; i >= 0; --i) {
            cw[i] = rw % stream_wg(K, i);
            rw /= stream_wg(K, i);
        }
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const int lc = (lane / line_lstride(K, i)) % line_ext(K, i);
            cl[i] = cw[i] * line_ext(K, i) + lc;
            vbase += (cl[i] + 1) * stream_stride(K, i);
            sig += cl[i];
            sigw += cw[i] * line_ext(K, i);
        }
    }
    int32_t *const vb = V + vbase;

    int tnext = 0;
    if (tid == 0) tnext = atomicAdd(L.ticket, 1);
    int cached_prob = -1;
    bool cached_live = false;
    while (true) {
        if (tid == 0) {
            misc[0] = ld_volatile(L.err) != 0 ? 0x7fffffff : tnext;
            if ((int64_t)tnext < L.ntickets) tnext = atomicAdd(L.ticket, 1);
        }
        __syncthreads();  // also: the previous column's last reads of shared memory are done
        const int t = misc[0];
        __syncthreads();  // every thread has the ticket before thread 0 may take the next
        if ((int64_t)t >= L.ntickets) break;
        const uint64_t ent = L.order[t];
        const int pidx = (int)(ent >> 32);
        const ProblemDesc &P = L.probs[pidx];
        const int col = (int)(uint32_t)ent;  // super-block index
        if (pidx != cached_prob) {            // the encode step's verdict (fixed before the fill)
            cached_prob = pidx;
            cached_live = ld_volatile(&P.istat->status) == 0;
        }
        if (!cached_live) continue;  // a failed problem: its columns publish nothing and read nothing

        int sco[NA], o[NA];  // super-block coordinates, its first line's coordinates
        {
            unsigned rem = (unsigned)col;
#pragma unroll
            for (int j = 0; j < NA; ++j) {
                const unsigned gs = (unsigned)P.sgstride[j];
                sco[j] = (int)(rem / gs);
                rem -= (unsigned)sco[j] * gs;
                o[j] = sco[j] * stream_sb(K, j);
            }
        }
        const int A = P.A;
        const int32_t *__restrict__ tab = P.tab;
        const uint8_t *__restrict__ codes = P.codes;
        const int rho = P.rho[NA], lens = P.len[NA], cofs = P.cofs[NA];
        const int ZQ = P.lzq;
        const int nblk = ZQ / U;  // blocks of the sweep: rho + SMAX steps, rounded up
        const int epoch = L.epoch;
        const int tagout = (int64_t)t == L.withhold ? 0 : epoch;  // a withheld column publishes nothing valid
        const int64_t FB = (int64_t)NFL * ZQ;  // face entries per super-block
        unsigned long long *Fq = reinterpret_cast<unsigned long long *>(P.Q);
        unsigned long long *Fo = Fq + (int64_t)col * FB;

        // this warp's tile (line block) for the traceback, or none past the grid
        int64_t tile = 0;
        bool has_tile = true;
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const int g = sco[i] * stream_wg(K, i) + cw[i];
            has_tile = has_tile && g < P.G[i];
            tile += (int64_t)g * P.gstride[i];
        }

        // neighbour super-blocks, the pair-table rows' residue codes; every ring
        // slot starts as "no cell"
        for (int S = tid; S <= M; S += NT) {
            int n = col;
            bool in = true;
#pragma unroll
            for (int i = 0; i < NA; ++i)
                if ((S >> i) & 1) {
                    in = in && sco[i] > 0;
                    n -= (int)P.sgstride[i];
                }
            nb[S] = in ? n : -1;
        }
        if (tid < NROW) {
            int x = 0, len = 0, cof = 0, row = 0;
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                if (tid >= row && tid < row + stream_sb(K, i)) {
                    x = o[i] + tid - row;
                    len = P.len[i];
                    cof = P.cofs[i];
                }
                row += stream_sb(K, i);
            }
            crow[tid] = (x >= 1 && x <= len) ? codes[cof + x - 1] : 0;
        }
        for (int i = tid; i < LY::PT; i += NT) V[i] = kNeg;
        if (tid < 7 + NX) misc[1 + tid] = 0;
        __syncthreads();  // nb, crow and the ring are read by every thread below

        if (tid >= NS) {
            // The exchanging warp. Chunk c of the halo is the consumer times [cU, cU + U):
            // four lanes per line load the producer's entries at those times + SB_S, 16 bytes
            // (two entries) each, again until both carry this launch's epoch, and store the
            // values into the ring (kNeg where there is no producer or its sweep does not
            // reach). A chunk may arrive once block c - 2 is swept; a swept block's faces go
            // out before anything else.
            const int q2 = lane % LQ, xw = (tid - NS) >> 5, sub = lane / LQ + LG * xw;
            // (each warp's own lines: those with j / LG mod NX = xw)
            for (int j = lane % LG + LG * xw; j < NH; j += LG * NX) {
                const uint32_t e = htab[j];
                const int src = nb[(e >> 21) & 31];
                hsrc[j] = src < 0 ? -1 : src * NFL + (int)((e >> 14) & 127);
            }
            __syncwarp();
            int out = 0, chunk = -1, batch = 0, tables = -2;  // next block out, next chunk and batch in
            uint64_t t0 = 0;
            for (int polls = 0; out < nblk;) {
                const int done = ld_acquire_shared(swept);
                bool moved = false;
                if (done > out) {  // face times [out U, out U + U) of the upper-face lines
                    const int sl = out % 3 * U + 2 * q2, tt = out * U + 2 * q2;
                    for (int f = sub; f < NFL; f += LG * NX) {
                        const int32_t *v = V + ftab[f] + sl;
                        st_relaxed_v2(Fo + (int64_t)f * ZQ + tt, tagged(v[0], tagout), tagged(v[1], tagout));
                    }
                    ++out;
                    moved = true;
                } else if (chunk < nblk && done >= chunk - 1) {
                    ulonglong2 x[HB];
                    bool ok = true;
                    const int tc = chunk * U + 2 * q2;
#pragma unroll
                    for (int u = 0; u < HB; ++u) {
                        const int j = (batch * HB + u) * LG * NX + sub;
                        x[u] = make_ulonglong2(tagged(kNeg, epoch), tagged(kNeg, epoch));
                        if (j < NH) {
                            const int line = hsrc[j], tp = tc + (int)(htab[j] >> 26);
                            if (line >= 0 && (unsigned)tp < (unsigned)ZQ)
                                x[u] = ld_relaxed_v2(Fq + (int64_t)line * ZQ + tp);
                        }
                    }
                    if (tables < chunk) {  // meanwhile the pair tables of positions cU + 1 .. (c + 1) U
                        int pent[PQ];
#pragma unroll
                        for (int u = 0; u < PQ; ++u) {
                            const int it = tid - NS + 32 * NX * u, p = chunk * U + 1 + it % U;
                            pent[u] = it < NROW * U && p >= 1 && p <= lens ? codes[cofs + p - 1] : 0;
                        }
#pragma unroll
                        for (int u = 0; u < PQ; ++u) {
                            const int it = tid - NS + 32 * NX * u;
                            if (it < NROW * U) pent[u] = __ldg(tab + crow[it / U] * A + pent[u]);
                        }
#pragma unroll
                        for (int u = 0; u < PQ; ++u) {
                            const int it = tid - NS + 32 * NX * u, p = chunk * U + 1 + it % U;
                            if (it < NROW * U) {
                                PT[it / U * ZS + (p & (R - 1))] = pent[u];
                                PT[it / U * ZS + (p & (R - 1)) + R] = pent[u];
                            }
                        }
                        tables = chunk;
                    }
#pragma unroll
                    for (int u = 0; u < HB; ++u)
                        ok = ok && (int)(x[u].x >> 32) == epoch && (int)(x[u].y >> 32) == epoch;
                    if (__all_sync(kFull, ok)) {
                        const int sl = (chunk + 3) % 3 * U + 2 * q2;
#pragma unroll
                        for (int u = 0; u < HB; ++u) {
                            const int j = (batch * HB + u) * LG * NX + sub;
                            if (j < NH) {
                                int32_t *v = V + (htab[j] & 0x3FFF) + sl;
                                v[0] = (int)(unsigned)x[u].x;
                                v[1] = (int)(unsigned)x[u].y;
                            }
                        }
                        if (++batch == NBATCH) {
                            batch = 0;
                            ++chunk;
                            __syncwarp();
                            if (lane == 0) st_release_shared(landed + xw, chunk);  // chunks below this one
                        }
                        moved = true;
                    }
                }
                if (moved) {
                    polls = 0;
                    t0 = 0;
                    continue;
                }
                if ((++polls & 15) == 0) {
                    if (t0 == 0) t0 = global_ns();
                    if (__any_sync(kFull, misc[3] != 0 || ld_volatile(L.err) != 0 ||
                                              (int64_t)(global_ns() - t0) > L.spin_ns)) {
                        misc[3] = 1;
                        break;
                    }
                }
                __nanosleep(polls < 64 ? 32 : 128);
            }
        } else {
            int Sp[M + 1];
            {
                int cd[NA];
#pragma unroll
                for (int i = 0; i < NA; ++i) {
                    const int x = o[i] + cl[i];
                    cd[i] = (x >= 1 && x <= P.len[i]) ? codes[P.cofs[i] + x - 1] : 0;
                }
                Sp[0] = 0;
#pragma unroll
                for (int h = 0; h < NA; ++h) {
                    int Rs[1 << (NA - 1)];
                    Rs[0] = 0;
#pragma unroll
                    for (int r = 1; r < (1 << h); ++r) Rs[r] = Rs[r & (r - 1)] + __ldg(tab + cd[lowbit_c(r)] * A + cd[h]);
#pragma unroll
                    for (int r = 0; r < (1 << h); ++r) Sp[r | (1 << h)] = Sp[r] + Rs[r];
                }
            }
            // The sweep. The origin's lane starts from H(0) = 0 as its "previous
            // position", which makes its key 0 with no move.
            int Wl = -sig * (1 << NA);  // W(x) = Wl + t 2^NA at step t
#pragma unroll
            for (int i = 0; i < NA; ++i) Wl += (o[i] + cl[i]) << i;
            int32_t *ptrow[NA];
            {
                int row = 0;
#pragma unroll
                for (int i = 0; i < NA; ++i) {
                    ptrow[i] = PT + (row + cl[i]) * ZS;
                    row += stream_sb(K, i);
                }
            }
            int vself = col == 0 && tid == 0 ? 0 : kNeg;
            int next = vself;  // best move of the next position that advances the last axis
            uint8_t *tbw = P.tb + tile * P.tb_block + lane - sigw * 32;  // this warp's traceback rows, by step
            int32_t *cur = vb, *prev = vb + 2 * U;  // the ring's slots of this block and the one before
            bool go = false;                        // this block's chunk is in place
            for (int b = 0; b < nblk; ++b) {
                if (!go) {  // uniform over the sweep's warps
                    if (warp == 0) {
                        const bool r = stream_wait(landed, NX, b + 1, misc + 3, L.spin_ns);
                        if (lane == 0) misc[2] = r;
                    }
                    sweep_barrier<NS>();
                    if (!misc[2]) break;
                }
                const int Wb0 = Wl + b * U * (1 << NA);
                const int zp0 = (b * U - sig) & (R - 1);
                const int32_t *ptb[NA];
#pragma unroll
                for (int i = 0; i < NA; ++i) ptb[i] = ptrow[i] + zp0;
                auto steps = [&](auto check) {
                    constexpr bool CHECK = decltype(check)::value != 0;
#pragma unroll
                    for (int s = 0; s < U; ++s) {
                        const int ts = b * U + s;
                        // a warp none of whose lanes holds a cell at this step skips it (every
                        // thread still meets the step's one barrier)
                        if (!CHECK || (unsigned)(ts - sigw) < (unsigned)(rho + line_skew_max(K))) {
                            const bool act = !CHECK || (unsigned)(ts - sig) < (unsigned)rho;
                            int p[NA];  // pair scores of the next position
#pragma unroll
                            for (int i = 0; i < NA; ++i) p[i] = ptb[i][s + 1];
                            int acc0 = next, acc1 = kNeg;  // two independent max chains
                            const int F = fold_subsets<NA, 0>(
                                [&](auto m) {  // the predecessor line's value popc(m) times ago
                                    constexpr int q = popc_c(m.value), off = stream_move_off<K>(m.value);
                                    return (s >= q ? cur[s - q - off] : prev[s - q + U - off]) + Sp[m.value];
                                },
                                p, acc0, acc1);
                            const int acc_all = max(acc0, acc1);
                            const int tm = (Wb0 + s * (1 << NA) - acc_all) & MASKB;
                            const int val = acc_all + tm;
                            if (has_tile) tbw[s * 32] = (uint8_t)tm;
                            if (act) {
                                cur[s] = val;
                                vself = val;
                            }
                            next = max(F, vself);
                        }
                        if (s == U - 2 && warp == 0) {
                            const bool r = __all_sync(kFull, ld_acquire_shared(landed + lane % NX) >= b + 2);
                            if (lane == 0) misc[4 + (b & 1)] = r;
                        }
                        sweep_barrier<NS>();
                    }
                };
                // most blocks: every lane of the warp on a cell in every step (without the checks
                // 0.948 -> 0.898 ms on k4 DNA, a fifth of a step's instructions)
                if (b * U >= sigw + line_skew_max(K) && (b + 1) * U <= sigw + rho)
                    steps(IntC<0>{});
                else
                    steps(IntC<1>{});
                if (tid == 0) st_release_shared(swept, b + 1);
                go = misc[4 + (b & 1)] != 0;
                tbw += U * 32;
                prev = cur;
                cur = cur == vb + 2 * U ? vb : cur + U;
            }
        }
        __syncthreads();
        const bool ok = misc[3] == 0;
        if (!ok) {
            if (tid == 0) atomicCAS(L.err, 0, MSA_ETIMEOUT);
            break;
        }
        // the corner's key: position len of the line holding the far corner
        {
            bool corner = true;
#pragma unroll
            for (int i = 0; i < NA; ++i) corner = corner && o[i] + cl[i] == P.len[i];
            if (corner && tid < NS) *P.qcorner = V[vbase + (lens + sig) % (3 * U)];
        }
    }
}

template <int K>
cudaError_t stream_attributes() {
    static DeviceOnce once;
    return once.run([] {
        return cudaFuncSetAttribute(fill_lines_stream_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    stream_smem_bytes<K>());
    });
}

template <int K>
cudaError_t launch_stream(const LaunchDesc &L, int grid, cudaStream_t s) {
    cudaError_t e = stream_attributes<K>();
    if (e != cudaSuccess) return e;
    fill_lines_stream_kernel<K><<<grid, stream_cta_threads<K>(), stream_smem_bytes<K>(), s>>>(L);
    return cudaGetLastError();
}

template <int K>
int stream_ctas() {
    if (stream_attributes<K>() != cudaSuccess) return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fill_lines_stream_kernel<K>, stream_cta_threads<K>(),
                                                      stream_smem_bytes<K>()) != cudaSuccess)
        return 0;
    return n;
}

}  // namespace msadp
