// Exact search-space pruning on the device, the restriction of the search space
// the paper leaves for future work (section 6: search only the partitions where
// an optimal alignment can lie), by the bound of Carrillo and Lipman. An
// alignment's sum-of-pairs score is the sum of the scores of its pairwise
// projections (gap against gap scores 0, section 5.2), and the projection of an
// alignment through cell x passes through (x_i, x_j), so no alignment through x
// scores above
//     U(x) = sum_{i<j} fwd_ij[x_i][x_j] + bwd_ij[x_i][x_j],
// fwd_ij / bwd_ij being the optimal pairwise scores of the prefixes / suffixes
// (Eq. 1 on each pair). A tile's bound is the sum over pairs of the largest
// fwd + bwd over the tile's rectangle of the (i, j) plane, never below U(x) of
// any cell inside; a tile whose bound is below a lower bound L on the optimum
// (the score of any feasible alignment) holds no cell of any optimal alignment,
// nor any optimal predecessor of such a cell, so the fill may leave it out and
// the optimal alignment (with its tie-break) is unchanged.
//
// Kernels, in stream order after the encode step:
//   pair_tables_kernel   fwd and bwd of every pair, one CTA per pair and direction
//   block_max_kernel     per pair, the largest fwd + bwd of every tile rectangle
//   greedy_bound_kernel  L: the score of the alignment built from the origin by
//                        taking, at every cell, the move to the neighbour with the
//                        largest U (ties: lowest mask) -- a feasible alignment
//   tile_bounds_kernel   per tile, the sum of its rectangles' maxima; the tiles
//                        below L are flagged for the fill and counted
// Pair values and U fit in 32 bits where the encode step accepts the problem: each
// is the score of a set of pairwise alignments, within its score bound.
#include "device_common.cuh"

#include <type_traits>

namespace msadp {

namespace {

// Pair tables: a skewed wavefront, one CTA per pair and direction. A pass covers
// kPairRows rows, 32 kPairR of them per warp: lane l owns rows kPairR l .. of its
// warp's and fills column s - l of them, top to bottom, at the warp's step s; the
// row above its first one comes from lane l - 1 by a shuffle of the previous step's
// last row. Lane 0 takes it from the warp above, which runs two chunks of 32 steps
// ahead, so one CTA barrier per chunk is enough (for the first warp: from the
// previous pass, read back from the table). A chunk's values are laid out in shared
// memory and written 32 columns of a row at a time. What bounds it is the chain of
// nb + 64 warps steps; with a thread per row, a barrier per step and every cell
// stored by itself (a store instruction touched as many lines as it has lanes) it
// took 0.69 ms for 700 / 760 / 800; now 0.27 ms.
constexpr int kPairR = 4;
constexpr int kPairWarps = 8;
constexpr int kPairRows = kPairR * 32 * kPairWarps;
constexpr int kPairStage = 33;  // ints per staged row (32 columns, one pad: conflict-free both ways)
constexpr int kPairEdge = 128;  // columns of a warp's last row kept for the warp below
constexpr int kPairMaxB = 16384;
constexpr int kPairSmem = kPairRows * kPairStage * 4 + (kPairWarps + 1) * kPairEdge * 4 + kPairMaxB;

__global__ void __launch_bounds__(kPairWarps * 32) pair_tables_kernel(const PruneDesc D) {
    const int pr = blockIdx.x;
    const bool rev = blockIdx.y != 0;  // false: prefixes (fwd), true: suffixes (bwd)
    const int i = D.pi[pr], j = D.pj[pr];
    const int na = D.len[i], nb = D.len[j], A = D.A, gap = D.gap;
    const uint8_t *a = D.codes + D.cofs[i], *b = D.codes + D.cofs[j];
    const int64_t W = (int64_t)nb + 1;
    // For the suffixes the same recurrence runs on the reversed sequences:
    // bwd[p][q] is the value at reversed coordinates (na - p, nb - q).
    int32_t *T = D.tables + D.toff[pr] + (rev ? 2 * ((int64_t)na + 1) * W - 1 : 0);
    const int64_t dp = rev ? -W : W, dq = rev ? -1 : 1;  // cell (p, q) at T + p dp + q dq
    extern __shared__ int32_t stage[];
    int32_t *edges = stage + kPairRows * kPairStage;
    uint8_t *cb = reinterpret_cast<uint8_t *>(edges + (kPairWarps + 1) * kPairEdge);  // code consumed at column q: cb[q]
    __shared__ int sub[MSA_MAX_ALPHABET * MSA_MAX_ALPHABET];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int32_t *mine = stage + w * 32 * kPairR * kPairStage;  // row r of lane l at (32 r + l) kPairStage
    int32_t *above = edges + w * kPairEdge, *below = above + kPairEdge;
    for (int c = t; c < A * A; c += kPairWarps * 32) sub[c] = D.sub[c];
    for (int q = t; q <= nb; q += kPairWarps * 32) cb[q] = q >= 1 ? (rev ? b[nb - q] : b[q - 1]) : 0;
    for (int p0 = 0; p0 <= na; p0 += kPairRows) {
        const int wrow = p0 + w * 32 * kPairR;  // this warp's first row
        const int p = wrow + lane * kPairR;
        const int nw = min(kPairWarps, (na - p0) / (32 * kPairR) + 1);  // warps with rows
        const int chunks = (nb + 1 + 31 + 31) / 32;                    // of a warp's steps
        int code[kPairR], left[kPairR];
#pragma unroll
        for (int r = 0; r < kPairR; ++r) {
            const int row = p + r;
            code[r] = row >= 1 && row <= na ? (rev ? a[na - row] : a[row - 1]) * A : 0;
            left[r] = 0;
        }
        int last = 0;   // this lane's last row at its previous column
        int diag0 = 0;  // the row above at the previous column
        __syncthreads();
        for (int ph = 0; ph < chunks + 2 * (nw - 1); ++ph) {
            const int c = ph - 2 * w;
            if (w < nw && c >= 0 && c < chunks) {  // uniform in the warp
                if (w == 0 && p0 > 0) {
                    const int q = 32 * c + lane;
                    if (q <= nb) above[q & (kPairEdge - 1)] = T[(p0 - 1) * dp + q * dq];
                    __syncwarp();
                }
                // every lane on a column >= 1: no checks (rows past the table are computed, not written)
                const bool inner = c >= 1 && 32 * c + 31 <= nb;
                auto step = [&](int k, auto check) {
                    constexpr bool CHECK = decltype(check)::value;
                    const int q = 32 * c + k - lane;
                    const int edge = above[(32 * c + k) & (kPairEdge - 1)];
                    int up = __shfl_up_sync(kFull, last, 1);
                    if (lane == 0) up = edge;
                    const bool on = !CHECK || (q >= 0 && q <= nb);
                    const int *tr = sub + cb[CHECK ? min(max(q, 0), nb) : q];
                    int v = up, d = diag0;
#pragma unroll
                    for (int r = 0; r < kPairR; ++r) {
                        // the column to the left and the diagonal first: only one add-max per row is chained
                        int x = max(left[r] + gap, d + tr[code[r]]);
                        if (CHECK && q <= 0) x = INT32_MIN;
                        if (p + r == 0) x = q <= 0 ? 0 : left[r] + gap;  // row 0 has no cell above
                        d = left[r];
                        v = p + r == 0 ? x : __viaddmax_s32(v, gap, x);
                        if (on) left[r] = v;
                        mine[(32 * r + lane) * kPairStage + k] = v;
                    }
                    if (on) {
                        last = v;
                        diag0 = up;
                        if (lane == 31) below[q & (kPairEdge - 1)] = v;
                    }
                };
                // the warp's rows, 32 columns each: row r of lane l holds columns 32 c - l ..
                auto flush = [&](auto check) {
                    constexpr bool CHECK = decltype(check)::value;
#pragma unroll
                    for (int r = 0; r < kPairR; ++r) {
                        int32_t *dst = T + (wrow + r) * dp + (32 * c + lane) * dq;
#pragma unroll 8
                        for (int l = 0; l < 32; ++l, dst += kPairR * dp - dq) {
                            const int q = 32 * c + lane - l;
                            const int v = mine[(32 * r + l) * kPairStage + lane];
                            if (!CHECK || (wrow + l * kPairR + r <= na && q >= 0 && q <= nb)) *dst = v;
                        }
                    }
                };
                if (inner) {
#pragma unroll 4
                    for (int k = 0; k < 32; ++k) step(k, std::false_type{});
                    __syncwarp();
                    if (wrow + 32 * kPairR - 1 <= na) flush(std::false_type{});
                    else flush(std::true_type{});
                } else {
#pragma unroll 1
                    for (int k = 0; k < 32; ++k) step(k, std::true_type{});
                    __syncwarp();
                    flush(std::true_type{});
                }
            }
            __syncthreads();
        }
    }
}

__device__ __forceinline__ int64_t pair_fb(const PruneDesc &D, int pr, int p, int q) {
    const int nb = D.len[D.pj[pr]];
    const int64_t W = (int64_t)nb + 1, n = ((int64_t)D.len[D.pi[pr]] + 1) * W;
    const int32_t *T = D.tables + D.toff[pr];
    return (int64_t)T[(int64_t)p * W + q] + T[n + (int64_t)p * W + q];
}

__global__ void block_max_kernel(const PruneDesc D) {
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < D.nblocks; g += (int64_t)gridDim.x * blockDim.x) {
        int pr = 0;
        while (pr + 1 < D.npairs && D.boff[pr + 1] <= g) ++pr;
        const int i = D.pi[pr], j = D.pj[pr];
        const int64_t r = g - D.boff[pr];
        const int bi = (int)(r / D.G[j]), bj = (int)(r - (int64_t)bi * D.G[j]);
        const int p0 = bi * D.E[i], p1 = min(p0 + D.E[i], D.len[i] + 1);
        const int q0 = bj * D.E[j], q1 = min(q0 + D.E[j], D.len[j] + 1);
        int64_t best = INT64_MIN / 4;
        for (int p = p0; p < p1; ++p)
            for (int q = q0; q < q1; ++q) best = max(best, pair_fb(D, pr, p, q));
        D.blk[g] = best;
    }
}

// The greedy walk. Its chain is one cell after another, so the pair sums it can
// meet are staged: the box of D + 1 coordinates per axis from the current cell, one
// (D + 1)^2 square of fwd + bwd per pair, and the residues; warp 0 walks until a
// coordinate leaves the box. Lanes judge a mask each (32 per round): the largest U,
// then the lowest mask win. One warp alone pays some 5 cycles per instruction, so a
// step only moves addresses and records its mask; the columns' scores follow per
// box, a lane per column. (700 / 760 / 800, 850 columns: 0.14 ms; from the tables in
// global memory, a column's score in its step, 2.35 ms.)
constexpr int kGreedyThreads = 1024;
__host__ __device__ constexpr int greedy_box(int K) { return K <= 5 ? 64 : K <= 7 ? 48 : 32; }
__host__ __device__ constexpr int greedy_smem(int K) {
    return K * (K - 1) / 2 * greedy_box(K) * greedy_box(K) * 4;
}

template <int K>
__global__ void __launch_bounds__(kGreedyThreads) greedy_bound_kernel(const PruneDesc D) {
    constexpr int B = greedy_box(K), NM = 1 << K, NP = K * (K - 1) / 2, NR = NM <= 32 ? 1 : NM / 32;
    extern __shared__ int32_t box[];
    __shared__ int sub[MSA_MAX_ALPHABET * MSA_MAX_ALPHABET];
    __shared__ uint8_t res[K][B];  // residue a move into coordinate lo + c consumes
    __shared__ uint8_t path[K * B];  // a box's columns
    __shared__ int at[K];
    __shared__ int state;          // 1: walk on, 0: at the corner or over the step limit
    const int tid = threadIdx.x, lane = tid & 31, A = D.A, gap = D.gap;
    for (int c = tid; c < A * A; c += kGreedyThreads) sub[c] = D.sub[c];
    if (tid < K) at[tid] = 0;
    if (tid == 0) state = 1;
    int64_t score = 0;  // of this lane's columns
    int steps = 0;
    __syncthreads();
    while (state) {
        int lo[K];
#pragma unroll
        for (int i = 0; i < K; ++i) lo[i] = at[i];
        {
            int pr = 0;
#pragma unroll
            for (int i = 0; i < K; ++i)
#pragma unroll
                for (int j = i + 1; j < K; ++j, ++pr) {
                    const int64_t W = (int64_t)D.len[j] + 1, n = ((int64_t)D.len[i] + 1) * W;
                    const int32_t *T = D.tables + D.toff[pr];
#pragma unroll 4
                    for (int c = tid; c < B * B; c += kGreedyThreads) {
                        const int p = lo[i] + c / B, q = lo[j] + c % B;
                        if (p <= D.len[i] && q <= D.len[j])
                            box[pr * B * B + c] = T[(int64_t)p * W + q] + T[n + (int64_t)p * W + q];
                    }
                }
        }
        if (tid < B)
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const int v = lo[i] + tid;
                res[i][tid] = v >= 1 && v <= D.len[i] ? D.codes[D.cofs[i] + v - 1] : 0;
            }
        __syncthreads();
        if (tid < 32) {
            int room[K], left[K];  // coordinates left to the end of the axis, and to the box's
            const int *cell[NR][NP];  // per round, this lane's entry of each pair's square
#pragma unroll
            for (int i = 0; i < K; ++i) {
                room[i] = D.len[i] - lo[i];
                left[i] = B - 1;
            }
#pragma unroll
            for (int w = 0; w < NR; ++w) {
                int p = 0;
#pragma unroll
                for (int i = 0; i < K; ++i)
#pragma unroll
                    for (int j = i + 1; j < K; ++j, ++p) {
                        const int m = 32 * w + lane;
                        cell[w][p] = box + p * B * B + (m >> i & 1) * B + (m >> j & 1);
                    }
            }
            int n = 0;
            bool corner = false, inside = true;
            while (inside) {
                int open = 0;
#pragma unroll
                for (int i = 0; i < K; ++i) open |= (room[i] > 0) << i;
                corner = open == 0;
                if (corner || steps > D.len_sum) break;
                int best = INT32_MIN, m = 0;
#pragma unroll
                for (int w = 0; w < NR; ++w) {
                    const int mm = 32 * w + lane;
                    int u = 0;
#pragma unroll
                    for (int p = 0; p < NP; ++p) u += *cell[w][p];
                    if (mm == 0 || mm >= NM || (mm & ~open) != 0) u = INT32_MIN;
                    const int top = __reduce_max_sync(kFull, u);
                    const int first = 32 * w + __ffs(__ballot_sync(kFull, u == top)) - 1;
                    if (top > best) {  // masks rise with the round: strict > keeps the lowest
                        best = top;
                        m = first;
                    }
                }
                int bit[K];
                inside = true;
#pragma unroll
                for (int i = 0; i < K; ++i) {
                    bit[i] = m >> i & 1;
                    room[i] -= bit[i];
                    left[i] -= bit[i];
                    inside = inside && left[i] > 0;
                }
                int p = 0;
#pragma unroll
                for (int i = 0; i < K; ++i)
#pragma unroll
                    for (int j = i + 1; j < K; ++j, ++p) {
                        const int d = bit[i] * B + bit[j];
#pragma unroll
                        for (int w = 0; w < NR; ++w) cell[w][p] += d;
                    }
                path[n] = (uint8_t)m;  // every lane the same byte
                ++n;
                ++steps;
            }
            __syncwarp();
            // the scores of the box's columns: a lane's coordinates are the moves up to its column
            int base[K];
#pragma unroll
            for (int i = 0; i < K; ++i) base[i] = 0;
            for (int c0 = 0; c0 < n; c0 += 32) {
                const int m = c0 + lane < n ? path[c0 + lane] : 0;
                int code[K];
#pragma unroll
                for (int i = 0; i < K; ++i) {
                    const unsigned moved = __ballot_sync(kFull, m >> i & 1);
                    code[i] = res[i][base[i] + __popc(moved & (0xffffffffu >> (31 - lane)))];
                    base[i] += __popc(moved);
                }
                int sp = gap * __popc(m) * (K - __popc(m));
#pragma unroll
                for (int i = 0; i < K; ++i)
#pragma unroll
                    for (int j = i + 1; j < K; ++j)
                        if ((m >> i) & (m >> j) & 1) sp += sub[code[i] * A + code[j]];
                score += sp;
            }
            if (lane == 0) {
#pragma unroll
                for (int i = 0; i < K; ++i) at[i] = lo[i] + base[i];
                state = !corner && steps <= D.len_sum;
            }
        }
        __syncthreads();
    }
    if (tid < 32) {
        for (int off = 16; off; off >>= 1) score += __shfl_xor_sync(kFull, score, off);
        if (lane == 0) *D.lower = score;
    }
}

template <int K>
cudaError_t launch_greedy(const PruneDesc &D, cudaStream_t s) {
    cudaError_t e =
        cudaFuncSetAttribute(greedy_bound_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, greedy_smem(K));
    if (e != cudaSuccess) return e;
    greedy_bound_kernel<K><<<1, kGreedyThreads, greedy_smem(K), s>>>(D);
    return cudaGetLastError();
}

__global__ void tile_bounds_kernel(const PruneDesc D) {
    const int64_t L = D.skip ? *D.lower : 0;
    unsigned long long tiles_out = 0, cells_out = 0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < D.ntiles; t += (int64_t)gridDim.x * blockDim.x) {
        int c[MSA_MAX_K];
        int64_t rem = t, cells = 1;
        for (int i = 0; i < D.k; ++i) {
            c[i] = (int)(rem / D.gstride[i]);
            rem -= (int64_t)c[i] * D.gstride[i];
            cells *= min(D.E[i], D.len[i] + 1 - c[i] * D.E[i]);
        }
        int64_t bound = 0;
        for (int pr = 0; pr < D.npairs; ++pr) bound += D.blk[D.boff[pr] + (int64_t)c[D.pi[pr]] * D.G[D.pj[pr]] + c[D.pj[pr]]];
        if (D.bound) D.bound[t] = bound;
        if (D.skip) {
            const bool out = bound < L;
            D.skip[t] = out;
            if (out) {
                ++tiles_out;
                cells_out += (unsigned long long)cells;
            }
        }
    }
    // one pair of atomics per block (one per tile left out was 0.17 ms for 250,000 tiles)
    if (D.skip) {
        __shared__ unsigned long long sum[2];
        if (threadIdx.x < 2) sum[threadIdx.x] = 0;
        __syncthreads();
        for (int off = 16; off; off >>= 1) {
            tiles_out += __shfl_xor_sync(kFull, tiles_out, off);
            cells_out += __shfl_xor_sync(kFull, cells_out, off);
        }
        if ((threadIdx.x & 31) == 0 && tiles_out) {
            atomicAdd(&sum[0], tiles_out);
            atomicAdd(&sum[1], cells_out);
        }
        __syncthreads();
        if (threadIdx.x < 2 && sum[threadIdx.x])
            atomicAdd(reinterpret_cast<unsigned long long *>(D.stats + threadIdx.x), sum[threadIdx.x]);
    }
}

}  // namespace

cudaError_t launch_prune(const PruneDesc &D, bool greedy, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(pair_tables_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem);
    if (e != cudaSuccess) return e;
    pair_tables_kernel<<<dim3(D.npairs, 2), kPairWarps * 32, kPairSmem, s>>>(D);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int64_t nbb = (D.nblocks + 255) / 256;
    block_max_kernel<<<(int)(nbb < 4096 ? (nbb < 1 ? 1 : nbb) : 4096), 256, 0, s>>>(D);
    e = cudaGetLastError();
    if (e == cudaSuccess && greedy)
        e = D.k == 2   ? launch_greedy<2>(D, s)
            : D.k == 3 ? launch_greedy<3>(D, s)
            : D.k == 4 ? launch_greedy<4>(D, s)
            : D.k == 5 ? launch_greedy<5>(D, s)
            : D.k == 6 ? launch_greedy<6>(D, s)
            : D.k == 7 ? launch_greedy<7>(D, s)
                       : launch_greedy<8>(D, s);
    if (e == cudaSuccess) {
        const int64_t nt = (D.ntiles + 255) / 256;
        tile_bounds_kernel<<<(int)(nt < 4096 ? (nt < 1 ? 1 : nt) : 4096), 256, 0, s>>>(D);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace msadp
