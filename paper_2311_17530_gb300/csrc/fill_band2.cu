// k = 2 band kernel: the pairwise DP (Eq. 1, section 2's 2^k - 1 = 3 neighbours
// for k = 2) as a skewed wavefront along warp lanes.
//
// A band is 32 R consecutive rows x0 of one problem; one warp fills it, lane l
// owning rows 32 R b + R l .. + R - 1 and sweeping the columns x1 four at a time, with
// a skew of one group of four columns per lane: at warp step t lane l fills its R x 4
// cells of columns 4 (t - l) .. + 3. The cells above its first row are lane l - 1's
// last row of the step before, so they arrive by four shuffles, issued as soon as
// that row exists; everything else is in the lane's registers. What bounds a single
// pair is the chain of steps (columns / 4 plus, per band, the skew and the handoff):
// inside a step the cells form a wavefront of R + 3 cells, two dependent instructions
// each, so a step of four columns costs little more than a step of one did. 5000 x 4800:
// 0.536 ms, against 1.214 ms one column per step (20 of a column step's 100
// instructions per cell, against 8).
//
// Lane 0 takes the cells above from the band above: its lane 31 lays its last row out
// in shared memory and every four steps the warp writes 16 columns of it to a face in
// global memory as (value, tag) 8-byte entries, the tag being the launch's epoch. The
// band below has the load of its next 16 entries in flight four steps before lane 0
// needs them and accepts them once every entry carries the epoch (a bounded wait), so
// no fence or release/acquire pair is needed: an aligned 8-byte entry is written by
// one store and read whole, and entries of earlier launches carry smaller epochs (the
// plan clears the faces before the first launch and when epochs wrap; serving clears
// them in the encode step). Bands are handed out by an atomic ticket in order, band
// above first, so a band only waits for a band already running.
//
// Values are the packed keys of every fill kernel without their W part,
// V = 4 (H - gap |x|), plus a tag per candidate: 2 for the cell above (mask 1), 1 for
// the cell to the left (mask 2), 0 for the diagonal (mask 3, plus the pair table entry
// ((sub - 2 gap) << 2)). One three-input max gives the best value and, in its low two
// bits, the tag of the lowest mask among ties. A cell is handed on with the tag of the
// move that will read it, V | 2 downwards and V | 1 to the right (the diagonal takes
// either: the table entries are lower by that tag), so one logic operation and one max
// are all there is between two cells. A mask is 3 - tag: a row's four tags are collected
// in a word, turned into masks by one complement and stored row-major. Columns past the
// last one (to the next multiple of 16, the tensor's row padding) are filled like any
// other and read by nobody.
#include "api_internal.h"
#include "device_common.cuh"

#include <type_traits>

namespace msadp {
namespace {

constexpr int R = kBand2RowsPerLane;
static_assert(R == 4, "a lane's pair-table entries of a column are one 16-byte load");
constexpr int kBandWarps = 2;   // warps per CTA, one band each (the tables take 16 KB a warp)
constexpr int kCodeRing = 256;  // columns whose residues are staged: 128 of skew, up to 128 ahead

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long *p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v));
}
__device__ __forceinline__ unsigned long long face_entry(int value, int tag) {
    return (unsigned long long)(unsigned)value | ((unsigned long long)(unsigned)tag << 32);
}

struct BandSmem {
    int4 tab[MSA_MAX_ALPHABET][32];  // pair-table entries of letter b with lane l's R rows
    int codes[kCodeRing];            // byte offset of a column's letter in tab
    int above[2][16];                // the band above's last row, two blocks of 16 columns
    int below[2][16];                // this band's
};

struct BandState {
    int left[R];   // this lane's rows at its previous column (V | 1)
    int up[4];     // the cells above its first row in the next step's columns (V | 2; lane 0: to be replaced)
    int diag;      // ... at the column before
    int t[4][R];   // pair-table entries of the next step's columns
    int4 code;     // codes of the step's after that
    int4 f;        // the band above's last row in the next step's columns
};

// Loads a step ahead: the next step's pair-table entries and the codes after those.
__device__ __forceinline__ void band_load(BandState &g, const BandSmem &sm, int lane, int grp) {
    const char *tab = reinterpret_cast<const char *>(&sm.tab[0][lane]);
    const int off[4] = {g.code.x, g.code.y, g.code.z, g.code.w};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int4 v = *reinterpret_cast<const int4 *>(tab + off[c]);
        g.t[c][0] = v.x, g.t[c][1] = v.y, g.t[c][2] = v.z, g.t[c][3] = v.w;
    }
    g.code = *reinterpret_cast<const int4 *>(&sm.codes[(4 * (grp + 1)) & (kCodeRing - 1)]);
}

// The R x 4 cells of a step, t the pair-table entries of its columns: their best
// candidates with tags and their masks by row; done(c, v) is told the last row's value
// of every column as soon as it exists. origin: the first cell is H(0) = 0, no move.
template <class Done>
__device__ __forceinline__ void band_tile(BandState &g, const int (&t)[4][R], const int (&up)[4], bool origin,
                                          uint32_t (&mask)[R], int (&acc)[R][4], const Done &done) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        int u = up[c], d = c ? up[c - 1] : g.diag;
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int diag = d + t[c][q];
            d = g.left[q];
            acc[q][c] = __vimax3_s32(u, g.left[q], diag);
            if (q == 0 && c == 0 && origin) acc[q][c] = 3;
            u = (acc[q][c] & ~3) | 2;
            g.left[q] = (acc[q][c] & ~3) | 1;
        }
        done(c, u);
    }
    g.diag = up[3];
#pragma unroll
    for (int q = 0; q < R; ++q)
        mask[q] = ~__byte_perm(__byte_perm((unsigned)acc[q][0], (unsigned)acc[q][1], 0x0040),
                               __byte_perm((unsigned)acc[q][2], (unsigned)acc[q][3], 0x0040), 0x5410) &
                  0x03030303u;
}

// KEEP: every cell's best candidate, V plus tag, is kept for the near-optimal walk, by
// step, row of the lane and lane (band2_kept_term): each 16-byte store of a warp is one
// run (row-major, a line per lane, 5000 x 4800 took 1.83 against 0.69 ms; the fill without
// KEEP 0.54).
template <bool KEEP>
__global__ void __launch_bounds__(kBandWarps * 32) fill_band2_kernel(const LaunchDesc L) {
    __shared__ BandSmem sms[kBandWarps];
    const int lane = threadIdx.x & 31;
    BandSmem &sm = sms[threadIdx.x >> 5];
    const int epoch = L.epoch;
    while (true) {
        int tk = 0, err = 0;
        if (lane == 0) {
            tk = atomicAdd(L.ticket, 1);
            err = ld_volatile(L.err);
        }
        tk = __shfl_sync(kFull, tk, 0);
        err = __shfl_sync(kFull, err, 0);
        if ((int64_t)tk >= L.ntickets || err != 0) break;
        const uint64_t ent = L.order[tk];
        const ProblemDesc &P = L.probs[(int)(ent >> 32)];
        const int band = (int)(uint32_t)ent;
        int st = 0;
        if (lane == 0) st = ld_volatile(&P.istat->status);
        // a failed problem: none of its bands works, so none waits for this one
        if (__shfl_sync(kFull, st, 0) != 0) continue;
        const int rho0 = P.rho[0], rho1 = P.rho[1];
        const int tagout = (int64_t)tk == L.withhold ? 0 : epoch;  // a withheld band publishes nothing valid
        const int64_t fstride = P.face0_stride / 2;                 // 8-byte entries per face
        unsigned long long *Fq = reinterpret_cast<unsigned long long *>(P.Q);
        const unsigned long long *face_in = Fq + (int64_t)(band - 1) * fstride;  // read for band > 0 only
        unsigned long long *face_out = Fq + (int64_t)band * fstride;
        const int i0 = band * 32 * R + lane * R;  // this lane's first row x0
        const uint8_t *c1 = P.codes + P.cofs[1];
        const int A = P.A;
        const int NG = (rho1 + 15) / 16 * 4;  // groups of four columns, whole blocks of 16
        __syncwarp();
        {
            const int *row[R];
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const int i = i0 + q;
                row[q] = P.tab + ((i >= 1 && i < rho0) ? (int)P.codes[P.cofs[0] + i - 1] * A : 0);
            }
            for (int b = 0; b < A; ++b)
                // for its diagonal, row 0 reads a cell handed down (V | 2), the others one handed right (V | 1)
                sm.tab[b][lane] = make_int4(__ldg(row[0] + b) - 2, __ldg(row[1] + b) - 1, __ldg(row[2] + b) - 1,
                                            __ldg(row[3] + b) - 1);
        }
        // column j consumes residue j - 1
        auto code_at = [&](int j) { return j >= 1 && j < rho1 ? (int)c1[j - 1] * (int)sizeof(sm.tab[0]) : 0; };
        // (every slot holds a letter: lanes before their first group load with it, unused)
        for (int j = lane; j < kCodeRing; j += 32) sm.codes[j] = code_at(j);
        if (lane < 16) sm.above[0][lane] = sm.above[1][lane] = kNeg | 2;
        int cnext = code_at(128 + lane);  // the 32 columns staged at step 8
        uint8_t *tbp[R];
#pragma unroll
        for (int q = 0; q < R; ++q)
            tbp[q] = P.tb + (int64_t)(i0 + q < rho0 ? i0 + q : 0) * P.tbstride[0] - 4 * lane;  // + 4 t: this lane's group
        int *kept = KEEP ? P.kept + (int64_t)band * band2_kept_steps(rho1) * (128 * R) + lane * 4 : nullptr;
        auto keep = [&](int q, int t, const int (&v)[4]) {
            *reinterpret_cast<int4 *>(kept + (int64_t)t * (128 * R) + q * 128) = make_int4(v[0], v[1], v[2], v[3]);
        };
        bool row_in[R];
#pragma unroll
        for (int q = 0; q < R; ++q) row_in[q] = i0 + q < rho0;
        const int gc = (rho1 - 1) >> 2;                                  // the far corner's group,
        const int qc = rho0 - 1 - i0;                                    // row
        const bool corner_lane = qc >= 0 && qc < R;

        BandState g;
#pragma unroll
        for (int q = 0; q < R; ++q) g.left[q] = kNeg | 1;
#pragma unroll
        for (int c = 0; c < 4; ++c) g.up[c] = kNeg | 2;
        g.diag = kNeg | 2;
        bool ok = true;
        unsigned long long e = 0;  // lane c < 16: the face entry of column c of the next block
        const bool taker = band > 0 && lane < 16;
        if (taker) e = ld_relaxed_u64(face_in + lane);
        __syncwarp();
        g.code = *reinterpret_cast<const int4 *>(&sm.codes[(-4 * lane) & (kCodeRing - 1)]);
        band_load(g, sm, lane, -lane);

        // Four steps from t0 (a multiple of 4). CHECK: some lane may be off its groups
        // [0, NG), or on the far corner's.
        auto block = [&](int t0, auto check) {
            constexpr bool CHECK = decltype(check)::value;
            const int blk = t0 >> 2;
            if (band > 0 && t0 < NG) {  // lane 0 enters the block's 16 columns
                uint64_t w0 = 0;
                for (int polls = 0; !__all_sync(kFull, lane >= 16 || (int)(e >> 32) == epoch); ++polls) {
                    if ((polls & 7) == 7) {
                        int expired = 0;
                        if (lane == 0) {
                            if (w0 == 0) w0 = global_ns();
                            expired = ld_volatile(L.err) != 0 || (int64_t)(global_ns() - w0) > L.spin_ns;
                        }
                        if (__shfl_sync(kFull, expired, 0)) {
                            ok = false;
                            return;
                        }
                        __nanosleep(polls < 64 ? 32 : 256);
                    }
                    if (taker) e = ld_relaxed_u64(face_in + 4 * t0 + lane);
                }
                if (lane < 16) sm.above[blk & 1][lane] = (int)(unsigned)e;
                if (taker && t0 + 4 < NG) e = ld_relaxed_u64(face_in + 4 * t0 + 16 + lane);
            }
            if ((t0 & 7) == 0 && t0 > 0) {
                // 32 more codes, columns 4 t0 + 96 .. + 127: they replace columns below
                // 4 t0 - 128, lane 31 reads from 4 t0 - 124 on
                sm.codes[(4 * t0 + 96 + lane) & (kCodeRing - 1)] = cnext;
                cnext = code_at(4 * t0 + 128 + lane);
            }
            __syncwarp();
            const int *above = sm.above[blk & 1];
            g.f = *reinterpret_cast<const int4 *>(above);
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const int t = t0 + s, grp = t - lane;
                const int up[4] = {lane == 0 ? g.f.x : g.up[0], lane == 0 ? g.f.y : g.up[1],
                                   lane == 0 ? g.f.z : g.up[2], lane == 0 ? g.f.w : g.up[3]};
                int te[4][R];
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int q = 0; q < R; ++q) te[c][q] = g.t[c][q];
                band_load(g, sm, lane, grp + 1);
                if (s < 3) g.f = *reinterpret_cast<const int4 *>(above + 4 * (s + 1));
                uint32_t mask[R];
                int acc[R][4], last[4];
                if constexpr (CHECK) {
                    // lanes off their groups hand down no cell (a branch around the tile: computing
                    // on and dropping the result was 3 % slower)
#pragma unroll
                    for (int c = 0; c < 4; ++c) last[c] = kNeg | 2;
                    if ((unsigned)grp < (unsigned)NG) {
                        band_tile(g, te, up, t == 0 && band == 0, mask, acc, [&](int c, int v) { last[c] = v; });
#pragma unroll
                        for (int q = 0; q < R; ++q)
                            if (row_in[q]) {
                                *reinterpret_cast<uint32_t *>(tbp[q] + 4 * s) = mask[q];
                                if constexpr (KEEP) keep(q, t, acc[q]);
                            }
                        if (grp == gc && corner_lane) {
                            int v = 0;  // a select chain: an index would put the registers in memory
#pragma unroll
                            for (int q = 0; q < R; ++q)
#pragma unroll
                                for (int c = 0; c < 4; ++c)
                                    if (q == qc && c == ((rho1 - 1) & 3)) v = acc[q][c] & ~3;
                            *P.qcorner = v + P.w_corner;
                        }
                    }
#pragma unroll
                    for (int c = 0; c < 4; ++c) g.up[c] = __shfl_up_sync(kFull, last[c], 1);
                } else {
                    band_tile(g, te, up, false, mask, acc, [&](int c, int v) {
                        last[c] = v;
                        g.up[c] = __shfl_up_sync(kFull, v, 1);
                    });
#pragma unroll
                    for (int q = 0; q < R; ++q)
                        if (row_in[q]) {
                            *reinterpret_cast<uint32_t *>(tbp[q] + 4 * s) = mask[q];
                            if constexpr (KEEP) keep(q, t, acc[q]);
                        }
                }
                if (lane == 31) *reinterpret_cast<int4 *>(&sm.below[((t - 31) >> 2) & 1][4 * ((t - 31) & 3)]) =
                    make_int4(last[0], last[1], last[2], last[3]);
                if (s == 2) {  // lane 31 has completed a block of 16 columns
                    __syncwarp();
                    const int ob = (t - 34) >> 2;  // its block
                    if (ob >= 0 && 4 * ob < NG && lane < 16)
                        st_relaxed_u64(face_out + 16 * ob + lane, face_entry(sm.below[ob & 1][lane], tagout));
                }
            }
#pragma unroll
            for (int q = 0; q < R; ++q) tbp[q] += 16;
        };
        int t0 = 0;
        for (; t0 < 32 && t0 < NG + 31 && ok; t0 += 4) block(t0, std::true_type{});
        for (; t0 + 3 < NG - 4 && ok; t0 += 4) block(t0, std::false_type{});
        for (; t0 < NG + 31 && ok; t0 += 4) block(t0, std::true_type{});
        if (!ok) {
            if (lane == 0) atomicCAS(L.err, 0, MSA_ETIMEOUT);
            break;
        }
    }
}

}  // namespace

cudaError_t launch_fill_band2(const LaunchDesc &L, int grid, cudaStream_t s) {
    if (L.keep)
        fill_band2_kernel<true><<<grid, kBandWarps * 32, 0, s>>>(L);
    else
        fill_band2_kernel<false><<<grid, kBandWarps * 32, 0, s>>>(L);
    return cudaGetLastError();
}

int fill_band2_ctas_per_sm() {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fill_band2_kernel<false>, kBandWarps * 32, 0) != cudaSuccess)
        return 0;
    return n;
}

int fill_band2_warps_per_cta() { return kBandWarps; }

}  // namespace msadp
