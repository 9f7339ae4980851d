// Whole-column super-block fill for k = 6 .. 8 with a short last axis (rho_s <= Z):
// the line kernel's sweep (fill_lines.cuh: lane l of a warp owns one line of a
// 32-line block, skewed by the sum of its local coordinates) on the streamed
// kernel's super-blocks (fill_lines_stream.cuh: a CTA of 4 warps owns 128 lines --
// 4 x 4 x 2 x 2 x 2, 2 x 4 x 2 x 2 x 2 x 2, 2^7 -- and sweeps them in lockstep, one
// barrier per step), with the halo exchanged as plain values once per column:
//
// * The cell update is the shared fold (fold_subsets): one load, one add where a
//   subset has pairs, one fused add-max and half a three-input maximum per subset,
//   only the result carried to the next position. Carrying every candidate instead
//   was 4.88 against 4.39 ms (k6 protein, 18 - 24 residues).
// * Shared memory holds the halo'd super-block (local coordinates -1 .. SB_i - 1)
//   indexed by POSITION: line h at word sum_i h_i A_i, its position z at word
//   + z + 1 (word 0 is position -1, "no cell"). At step t lane c reads position
//   t - sigma(c) of its predecessor lines; the 32 lanes of a warp hit 32 banks
//   when sum_i c_i (A_i - 1) is distinct mod 32 over a line block (strides found
//   by exhaustive search, footprint within 1 % of the unpadded box).
// * A column waits for the completion flags of its face neighbours along the
//   line axes (their own waits make the diagonal neighbours complete as well),
//   loads its halo lines (547 at k = 6) from their producers' faces, sweeps
//   rho_s + SMAX steps, writes its upper-face lines back, and publishes its flag with
//   a release store after a CTA barrier. Per halo value that is a quarter of a
//   16-byte load and one shared store, against a tagged 8-byte entry, its check and
//   its ring store per value in the pipelined form; a column cannot start before its
//   producers have finished theirs, which on a last axis of 25 positions costs
//   less than the per-block exchange.
// * A face holds its lines side by side in groups of four positions: neighbouring
//   lanes load neighbouring lines, each thread a line, with the loads of two to five
//   lines in flight and the pair sums formed meanwhile. Line by line (consecutive
//   groups of a line on neighbouring lanes, stores to shared memory four words apart)
//   the halo took 22,000 of a column's 53,000 cycles, 16,000 now.
// * A ticket is a unit of one or more super-blocks along axis J = k - 2, filled one
//   after the other: the lines at h_J = SB_J become the next one's lines at h_J = 0
//   in shared memory, and the pair sums and tables without axis J stay (the planner's
//   wide_chain says when this pays).
//
// Measured (fill, against the form without the last two): 18 - 24 residues at k = 6
// 4.33 -> 3.67 ms, 8 each 0.163 -> 0.146; 9 - 12 at k = 7 1.26 -> 1.00; 8 each at k = 8
// 8.5 -> 5.5. A step is 184 issue cycles of a warp and 12 warps fill an SM, so a sweep
// is bound by the integer pipe while three CTAs sweep together (530 - 600 cycles a
// step); over a whole column it is at half of that rate, the rest being the halo's
// latency. A CTA barrier only every 2 / 4 / 8 steps, with the warps that many steps
// apart, was slower (4.42 / 4.51 / 4.74 at k = 6): the sweep gets longer.
//
// Global memory: the traceback bytes of each line block (layout 3 spanning the
// whole last axis, as the streamed kernel), the faces of each super-block: its
// upper-face lines by groups of four positions, rho_s rounded up to 4 of them.
#pragma once

#include "device_common.cuh"

namespace msadp {


// Strides (words) of the line axes in the position-indexed super-block box.
__host__ __device__ constexpr int wide_stride(int K, int i) {
    constexpr int k6[] = {26, 393, 131, 1965, 5905};
    constexpr int k7[] = {14, 42, 211, 633, 1901, 5713};
    constexpr int k8[] = {10, 30, 90, 271, 813, 2449, 7353};
    return K == 6 ? k6[i] : K == 7 ? k7[i] : k8[i];
}
template <int K>
__host__ __device__ constexpr int wide_move_off(int m) {
    int s = 0;
    for (int i = 0; i < K - 1; ++i)
        if ((m >> i) & 1) s += wide_stride(K, i);
    return s;
}
template <int K>
__host__ __device__ constexpr int wide_v_words() {
    // the last word any line's positions -1 .. Z - 1 use, plus one, plus the 3
    // words past the last position that a face write-back's last group reads
    int s = wide_z(K) + 1;
    for (int i = 0; i < K - 1; ++i) s += stream_sb(K, i) * wide_stride(K, i);
    return round_up(s + 3, 4);
}
template <int K>
struct WideLayout {
    static constexpr int NA = K - 1;
    static constexpr int NT = 32 * stream_warps(K);
    static constexpr int NHL = [] {
        int n = 1;
        for (int i = 0; i < K - 1; ++i) n *= stream_sb(K, i) + 1;
        return n;
    }();
    static constexpr int NH = NHL - NT;
    static constexpr int NFL = stream_face_lines(K);
    static constexpr int NROW = [] {
        int n = 0;
        for (int i = 0; i < K - 1; ++i) n += stream_sb(K, i);
        return n;
    }();
    // pair-table rows: positions 0 .. Z - 1, row stride congruent to a line
    // block's skew + 1 mod 32 (lanes of one row read different positions)
    static constexpr int ZS = [] {
        int s = wide_z(K);
        while (s % 32 != (line_skew_max(K) + 1) % 32) ++s;
        return s;
    }();
    static constexpr int PT = 0;
    static constexpr int HDESC = PT + round_up(NROW * ZS, 4);  // halo lines: base | face line << 15 | S << 22
    static constexpr int FTAB = HDESC + round_up(NH, 4);       // face lines: base
    static constexpr int NB = FTAB + round_up(NFL, 4);
    static constexpr int CROW = NB + round_up(1 << NA, 4);
    static constexpr int MISC = CROW + round_up(NROW, 4);
    static constexpr int V = MISC + 8;  // reads at most SMAX - 1 words below the box stay in the tables
    static constexpr int WORDS = V + wide_v_words<K>();
};
template <int K>
__host__ __device__ constexpr int wide_smem_bytes() {
    return WideLayout<K>::WORDS * 4;
}
template <int K>
__host__ __device__ constexpr int wide_min_ctas() {
    int c = (228 * 1024) / (wide_smem_bytes<K>() + 1024);
    return c < 1 ? 1 : c;
}

// SHORT: at most kWideShort positions a line, so that more lines' loads fit in flight
// (4^6 cells, four waves of super-blocks: 0.0270 against 0.0343 ms).
constexpr int kWideShort = 12;
template <int K, bool SHORT>
__global__ void __launch_bounds__(stream_threads<K>(), wide_min_ctas<K>()) fill_lines_wide_kernel(const LaunchDesc L) {
    using LY = WideLayout<K>;
    constexpr int NA = K - 1;
    constexpr int M = (1 << NA) - 1;
    constexpr int NT = LY::NT, NH = LY::NH, NHL = LY::NHL, NFL = LY::NFL, NROW = LY::NROW, ZS = LY::ZS;
    constexpr int SMAX = stream_skew_max(K);
    constexpr int MASKB = (1 << K) - 1;
    constexpr int NQM = ((SHORT ? kWideShort : wide_z(K)) + 3) / 4;  // groups of 4 positions of a line, at most
    constexpr int J = NA - 1, SBJ = stream_sb(K, J);  // the axis a unit of work runs along
    constexpr int NC = NHL / (SBJ + 1);            // lines with h_J = 0, all of them halo
    constexpr int CZ = wide_z(K) > 16 ? 32 : 16;   // lanes copying one line's positions
    constexpr int HB = NQM >= 7 ? 2 : NQM >= 4 ? 3 : 5;           // ... whose loads are in flight together
    static_assert(SMAX < LY::V && wide_v_words<K>() < (1 << 15) && NFL <= NT && NFL < 128 && NA < 10, "geometry");

    extern __shared__ __align__(16) unsigned char smem_raw[];
    int32_t *sm = reinterpret_cast<int32_t *>(smem_raw);
    int32_t *PT = sm + LY::PT;
    uint32_t *hdesc = reinterpret_cast<uint32_t *>(sm + LY::HDESC);
    int32_t *ftab = sm + LY::FTAB;
    int32_t *nb = sm + LY::NB;
    int32_t *crow = sm + LY::CROW;
    volatile int32_t *misc = sm + LY::MISC;  // [0] ticket, [1] wait verdict
    int32_t *V = sm + LY::V;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // Once per CTA: the face lines (some c_i = SB_i - 1) in line order with their
    // box bases, then every halo line (some digit h_i = 0) with its base, the
    // number of its producer's face line (c_i = SB_i - 1 where h_i = 0, h_i - 1
    // elsewhere) and the subset S of axes at -1 (which neighbour produces it).
    for (int j = tid; j < NT; j += NT) {
        int c[NA], base = 0;
        super_line<K>(j, c);
        const int f = face_number<K>(c);
#pragma unroll
        for (int i = 0; i < NA; ++i) base += (c[i] + 1) * wide_stride(K, i);
        if (f >= 0) ftab[f] = base;
    }
    // Position -1 of every line, which no column changes, is set here too.
    for (int j = tid; j < NHL; j += NT) {
        int rem = j, base = 0;
#pragma unroll
        for (int i = NA - 1; i >= 0; --i) {
            base += (rem % (stream_sb(K, i) + 1)) * wide_stride(K, i);
            rem /= stream_sb(K, i) + 1;
        }
        V[base] = kNeg;
    }
    for (int j = tid; j < NHL; j += NT) {
        int h[NA], c[NA], base = 0;
        uint32_t S = 0;
        int n = halo_number<K>(j, h);
        if (n < 0) continue;
        // the lines with h_J = 0 last (every SBJ + 1st line of the box)
        n = h[J] == 0 ? NH - NC + j / (SBJ + 1) : n - (j / (SBJ + 1) + 1);
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            base += h[i] * wide_stride(K, i);
            c[i] = h[i] == 0 ? stream_sb(K, i) - 1 : h[i] - 1;
            if (h[i] == 0) S |= 1u << i;
        }
        hdesc[n] = (uint32_t)base | (uint32_t)face_number<K>(c) << 15 | S << 22;
    }

    // this thread's line: warp and lane coordinates, box base, skew
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
            vbase += (cl[i] + 1) * wide_stride(K, i);
            sig += cl[i];
            sigw += cw[i] * line_ext(K, i);
        }
    }

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
        int col = (int)(uint32_t)ent;  // the unit's first super-block
        if (pidx != cached_prob) {
            cached_prob = pidx;
            cached_live = ld_volatile(&P.istat->status) == 0;
        }
        if (!cached_live) continue;  // a failed problem: its columns read and publish nothing

        int sco[NA], o[NA];
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
        const int rho = P.rho[NA], cofs = P.cofs[NA];
        const int ZQ = (rho + 3) & ~3;  // words per face line
        const int NQ = ZQ / 4;
        const int64_t FB = (int64_t)NFL * ZQ;
        const int32_t *Fq = P.Q;
        int32_t *const done = L.done + P.tile_base;

        // super-blocks of this unit: up to P.chain of them along axis J
        const int jend = min(sco[J] + P.chain, (P.G[J] + stream_wg(K, J) - 1) / stream_wg(K, J));
        int Sp[M + 1], cd[NA];
        bool first = true;
        while (true) {
            int32_t *Fo = P.Q + (int64_t)col * FB;
            const int nh = first ? NH : NH - NC;  // halo lines to load
            int64_t tile = 0;
            bool has_tile = true;
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                const int g = sco[i] * stream_wg(K, i) + cw[i];
                has_tile = has_tile && g < P.G[i];
                tile += (int64_t)g * P.gstride[i];
            }

            // neighbour super-blocks, pair-table rows' residue codes
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
            __syncthreads();  // nb and crow are read below
            // face neighbours along the line axes (one lane of warp 0 each; their completion
            // implies that of every diagonal neighbour), and meanwhile the pair tables of the
            // last axis against every line axis, positions 0 .. rho - 1
            if (warp == 0) {
                bool ok = true;
                if (lane < NA && sco[lane] > 0 && (first || lane != J))
                    ok = wait_at_least(done + nb[1 << lane], 1, L.err, L.spin_ns);
                ok = __all_sync(kFull, ok);
                if (lane == 0) misc[1] = ok;
            } else {
                for (int z = lane; z < rho; z += 32) {
                    const int cz = z >= 1 ? codes[cofs + z - 1] : 0;
                    for (int row = (first ? 0 : NROW - SBJ) + warp - 1; row < NROW; row += NT / 32 - 1)
                        PT[row * ZS + z] = __ldg(tab + crow[row] * A + cz);
                }
            }
            __syncthreads();  // the waiting lanes' acquires precede every thread's halo loads
            if (!misc[1]) {
                if (tid == 0) atomicCAS(L.err, 0, MSA_ETIMEOUT);
                return;
            }

            // The halo: positions 0 .. rho - 1 of every halo line, a line per thread and turn
            // (neighbouring lanes read neighbouring lines of one face, 16 bytes each), HB
            // lines' loads in flight; the first of them fly while the pair sums are formed.
            int4 hv[HB][NQM];
            int hdst[HB];
            auto halo_load = [&](int s0) {
#pragma unroll
                for (int u = 0; u < HB; ++u) {
                    const int j = (s0 + u) * NT + tid;
                    hdst[u] = -1;
                    if (j >= nh) continue;
                    const uint32_t e = hdesc[j];
                    const int src = nb[e >> 22];
                    hdst[u] = (int)(e & 0x7FFF) + 1;
                    const int4 *p = reinterpret_cast<const int4 *>(Fq + (int64_t)src * FB) + (int)((e >> 15) & 127);
#pragma unroll
                    for (int q = 0; q < NQM; ++q) {
                        hv[u][q] = make_int4(kNeg, kNeg, kNeg, kNeg);
                        if (src >= 0 && q < NQ) hv[u][q] = __ldcg(p + q * NFL);
                    }
                }
            };
            auto halo_store = [&]() {
#pragma unroll
                for (int u = 0; u < HB; ++u) {
                    if (hdst[u] < 0) continue;
                    int32_t *d = V + hdst[u];
#pragma unroll
                    for (int q = 0; q < NQM; ++q) {
                        if (4 * q < rho) d[4 * q] = hv[u][q].x;
                        if (4 * q + 1 < rho) d[4 * q + 1] = hv[u][q].y;
                        if (4 * q + 2 < rho) d[4 * q + 2] = hv[u][q].z;
                        if (4 * q + 3 < rho) d[4 * q + 3] = hv[u][q].w;
                    }
                }
            };
            halo_load(0);
            // this line's pair sums over subsets of the line axes; along the unit only
            // those with axis J change
            const int xj = o[J] + cl[J];
            const int cj = (xj >= 1 && xj <= P.len[J]) ? codes[P.cofs[J] + xj - 1] : 0;
            if (first) {
                Sp[0] = 0;
#pragma unroll
                for (int i = 0; i < J; ++i) {
                    const int x = o[i] + cl[i];
                    cd[i] = (x >= 1 && x <= P.len[i]) ? codes[P.cofs[i] + x - 1] : 0;
                }
#pragma unroll
                for (int h = 0; h < J; ++h) {
                    int Rs[1 << (NA - 1)];
                    Rs[0] = 0;
#pragma unroll
                    for (int r = 1; r < (1 << h); ++r) Rs[r] = Rs[r & (r - 1)] + __ldg(tab + cd[lowbit_c(r)] * A + cd[h]);
#pragma unroll
                    for (int r = 0; r < (1 << h); ++r) Sp[r | (1 << h)] = Sp[r] + Rs[r];
                }
            }
            {
                int Rs[1 << J];
                Rs[0] = 0;
#pragma unroll
                for (int r = 1; r < (1 << J); ++r) Rs[r] = Rs[r & (r - 1)] + __ldg(tab + cd[lowbit_c(r)] * A + cj);
#pragma unroll
                for (int r = 0; r < (1 << J); ++r) Sp[r | (1 << J)] = Sp[r] + Rs[r];
            }
            halo_store();
#pragma unroll 1
            for (int s0 = HB; s0 * NT < nh; s0 += HB) {
                halo_load(s0);
                halo_store();
            }
            __syncthreads();

            // The sweep: rho + SMAX steps, one barrier each. Every lane reads its own
            // skewed position, in range or not (a read below position -1 or past the
            // last position feeds only candidates that are overwritten or never
            // stored); the origin's lane starts from H(0) = 0 as its previous position.
            int Wl = -sig * (1 << NA);  // W(x) = Wl + t 2^NA at step t
#pragma unroll
            for (int i = 0; i < NA; ++i) Wl += (o[i] + cl[i]) << i;
            int ptoff[NA];
            {
                int row = 0;
#pragma unroll
                for (int i = 0; i < NA; ++i) {
                    ptoff[i] = (row + cl[i]) * ZS;
                    row += stream_sb(K, i);
                }
            }
            int vself = col == 0 && tid == 0 ? 0 : kNeg;
            int D = vself;  // best move of the next position that advances the last axis
            const int rows = P.tb_block / 32;
            uint8_t *tbw = P.tb + tile * P.tb_block + lane;
            const int nsteps = rho + SMAX;
            for (int ts = 0; ts < nsteps; ++ts) {
                if ((unsigned)(ts - sigw) < (unsigned)(rho + line_skew_max(K))) {
                    const int z = ts - sig;
                    const bool act = (unsigned)z < (unsigned)rho;
                    const int zn = z < -1 ? 0 : (z + 1 >= rho ? rho - 1 : z + 1);
                    int p[NA];
#pragma unroll
                    for (int i = 0; i < NA; ++i) p[i] = PT[ptoff[i] + zn];
                    int acc0 = D, acc1 = kNeg;
                    const int32_t *vp = V + vbase + z + 1;
                    const int F = fold_subsets<NA, 0>(
                        [&](auto m) { return vp[-wide_move_off<K>(m.value)] + Sp[m.value]; }, p, acc0, acc1);
                    const int acc = max(acc0, acc1);
                    const int tm = (Wl + ts * (1 << NA) - acc) & MASKB;
                    const int val = acc + tm;
                    const int r = ts - sigw;
                    if (has_tile && r < rows) tbw[(int64_t)r * 32] = (uint8_t)tm;
                    if (act) {
                        V[vbase + z + 1] = val;
                        vself = val;
                    }
                    D = max(F, vself);
                }
                __syncthreads();
            }

            // faces for the successors: every position of the upper-face lines
            if (tid < NFL) {
                const int32_t *v = V + ftab[tid] + 1;
                int4 *dst = reinterpret_cast<int4 *>(Fo) + tid;
                for (int q = 0; q < NQ; ++q, v += 4) dst[q * NFL] = make_int4(v[0], v[1], v[2], v[3]);
            }
            // the next super-block's lines with h_J = 0 are this one's with h_J = SB_J
            const bool more = sco[J] + 1 < jend;
            if (more)
                for (int m = tid / CZ; m < NC; m += NT / CZ) {
                    int32_t *to = V + (hdesc[NH - NC + m] & 0x7FFF) + 1;
                    const int z = tid % CZ;
                    if (z < rho) to[z] = to[SBJ * wide_stride(K, J) + z];
                }
            {
                bool corner = true;
#pragma unroll
                for (int i = 0; i < NA; ++i) corner = corner && o[i] + cl[i] == P.len[i];
                if (corner) *P.qcorner = V[vbase + rho];
            }
            __syncthreads();  // every thread's face stores precede the release
            if (tid == 0 && (int64_t)t != L.withhold) st_release(done + col, 1);
            if (!more) break;
            first = false;
            col += (int)P.sgstride[J];
            ++sco[J];
            o[J] += SBJ;
        }
    }
}

template <int K>
cudaError_t wide_attributes() {
    static DeviceOnce once;
    return once.run([] {
        cudaError_t e = cudaFuncSetAttribute(fill_lines_wide_kernel<K, true>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, wide_smem_bytes<K>());
        if (e == cudaSuccess && wide_z(K) > kWideShort)
            e = cudaFuncSetAttribute(fill_lines_wide_kernel<K, (wide_z(K) <= kWideShort)>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, wide_smem_bytes<K>());
        return e;
    });
}

template <int K>
cudaError_t launch_wide(const LaunchDesc &L, int grid, cudaStream_t s, int rho_s) {
    cudaError_t e = wide_attributes<K>();
    if (e != cudaSuccess) return e;
    if (rho_s <= kWideShort)
        fill_lines_wide_kernel<K, true><<<grid, stream_threads<K>(), wide_smem_bytes<K>(), s>>>(L);
    else
        fill_lines_wide_kernel<K, (wide_z(K) <= kWideShort)><<<grid, stream_threads<K>(), wide_smem_bytes<K>(), s>>>(L);
    return cudaGetLastError();
}

template <int K>
int wide_ctas() {
    if (wide_attributes<K>() != cudaSuccess) return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fill_lines_wide_kernel<K, (wide_z(K) <= kWideShort)>,
                                                      stream_threads<K>(), wide_smem_bytes<K>()) != cudaSuccess)
        return 0;
    return n;
}

}  // namespace msadp
