// Optimal and near-optimal alignments on the device (section 6 proposes
// retrieving further solutions by forking at equally ranked paths, or within a
// threshold the user sets): every alignment scoring at least OPT - delta,
// enumerated from the far corner by a depth-first walk over the kept score
// tensor, the moves of each column tried in increasing mask order (so the
// alignments come in increasing lexicographic order of their reversed column
// sequence, the first being the single-alignment traceback's for delta = 0).
//
// A move m from cell x to p = x - e_m is followed when
//     H(p) + SP(m at x) + (score of the columns already fixed) >= OPT - delta,
// H being the forward tensor: H(p) is the best any completion through p can add,
// so every qualifying alignment is reached and no other one is produced.
//
// The fill is the generic tile kernel, which keeps the packed key of every cell:
// Q(x) = H'(x) 2^k + W(x) with H'(x) = H(x) - gap (k - 1) |x|_1 and
// W(x) = sum_i 2^i x_i, so H(x) = (Q(x) - W(x)) / 2^k + gap (k - 1) |x|_1
// exactly (and in 32 bits: every sum compared below is the score of an alignment,
// which the encode step's range check keeps in range).
//
// One warp walks, and what bounds it is the chain of one node: residue codes and
// offsets from shared memory, one score per lane, a ballot. At a node every mask is
// judged at once, a lane per mask (and 32 masks per round), and the set that
// qualifies goes on the stack, so going back costs no judging: the lanes look 32
// depths at a time for the deepest one with a mask left and count the moves to undo
// with one ballot per axis. The offset of a cell is a sum of one term per axis in
// every layout of the scores, so the terms are tabulated per coordinate once.
// 256 alignments of 120 x 110 x 130 (9,100 moves followed): 24.6 ms when the walk
// went back one column at a time, judging again, with positions in local memory.
#include "device_common.cuh"

namespace msadp {

namespace {

constexpr int kNearThreads = 256;
constexpr int kNearSmem = 160 * 1024;  // tables and stack beyond this stay in global memory

// Term of coordinate v of axis i in the element offset of a cell's score: row-major
// (qstride) for k <= 3, tile-major (the traceback's layout 2) for k >= 4.
__device__ __forceinline__ int64_t axis_offset(const ProblemDesc &P, int i, int v) {
    if (P.tb_layout != 2) return (int64_t)v * P.qstride[i];
    const int q = v / P.E[i];
    return (int64_t)q * P.gstride[i] * P.tb_block + (int64_t)(v - q * P.E[i]) * P.lst[i];
}

__host__ __device__ constexpr int near_words(int K) { return K <= 5 ? 1 : 1 << (K - 5); }  // 32-mask rounds: lane l judges mask 32 w + l

// Bytes of the walk's tables and stack (8-byte terms, hit sets, scores, codes, moves).
size_t near_bytes(int k, int64_t len_sum) {
    const size_t depth = (size_t)len_sum + 1;
    return ((size_t)len_sum + k) * 8 + depth * 4 * near_words(k) + depth * 4 + (size_t)len_sum + 16 + depth + 64;
}

template <int K>
__global__ void __launch_bounds__(kNearThreads) near_optimal_kernel(const ProblemDesc *probs, IODesc io, int64_t delta,
                                                                    int32_t max_count, NearOut o, int in_smem) {
    constexpr int NW = near_words(K), NM = 1 << K, NP = K * (K - 1) / 2;
    extern __shared__ __align__(16) unsigned char near_smem[];
    __shared__ int sub[MSA_MAX_ALPHABET * MSA_MAX_ALPHABET];
    const ProblemDesc &P = probs[0];
    const int lane = threadIdx.x & 31;
    const int A = P.A, total = P.len_sum, depths = total + 1;
    if (ld_volatile(&P.istat->status) != 0) {  // the fill did not complete: nothing to enumerate
        if (threadIdx.x == 0) {
            o.count_more[0] = 0;
            o.count_more[1] = 0;
        }
        return;
    }
    // tables: per axis the offset term of every coordinate; the residue codes; the pair scores
    unsigned char *base = in_smem ? near_smem : o.work;
    int64_t *off = reinterpret_cast<int64_t *>(base);
    unsigned *hits = reinterpret_cast<unsigned *>(off + total + K);
    int *accs = reinterpret_cast<int *>(hits + (size_t)depths * NW);
    uint8_t *codes = reinterpret_cast<uint8_t *>(accs + depths);
    uint8_t *path = codes + ((total + 15) & ~15);
    int cofs[K], at[K];  // first code of sequence i, first entry of axis i in off
#pragma unroll
    for (int i = 0; i < K; ++i) {
        cofs[i] = P.cofs[i];
        at[i] = cofs[i] + i;
    }
#pragma unroll
    for (int i = 0; i < K; ++i)
        for (int v = threadIdx.x; v < P.rho[i]; v += kNearThreads) off[at[i] + v] = axis_offset(P, i, v);
    for (int c = threadIdx.x; c < total; c += kNearThreads) codes[c] = P.codes[c];
    for (int c = threadIdx.x; c < A * A; c += kNearThreads) sub[c] = io.subst[c];
    __syncthreads();
    if (threadIdx.x >= 32) return;

    const int gap = io.gap, u = gap * (K - 1);
    int x[K], S = 0, W = 0;
    int64_t corner = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        x[i] = P.len[i];
        S += x[i];
        W += x[i] << i;
        corner += off[at[i] + x[i]];
    }
    const int32_t *Q = P.Q;
    const int opt = ((Q[corner] - W) >> K) + u * S;
    // OPT - delta (no alignment scores below the 32-bit range)
    const int thr = delta > (int64_t)opt - INT32_MIN ? INT32_MIN : (int)(opt - delta);
    int d = 0, count = 0, more = 0;
    int acc = 0;  // score of the columns fixed so far (depth d)
    // Every move followed leads to at least one qualifying alignment (H(p) is
    // reached by some path), so at most total + 1 nodes are judged per alignment
    // stored, plus one walk; the bound below only guards that argument.
    const int64_t limit = ((int64_t)total + 1) * ((int64_t)max_count + 1) + 2;
    for (int64_t it = 0;; ++it) {
        if (it > limit) {
            more = 2;  // reported as an inconsistent tensor
            break;
        }
        if (S == 0) {
            __syncwarp();  // lane 0's moves
            uint8_t *dst = o.masks + (int64_t)count * total;
            for (int c = lane; c < d; c += 32) dst[c] = path[d - 1 - c];
            if (lane == 0) {
                o.ncols[count] = d;
                o.scores[count] = acc;
            }
            ++count;
        } else {
            // the pair scores of the residues at x and the axes that can still move
            int open = 0, code[K];
#pragma unroll
            for (int i = 0; i < K; ++i) {
                open |= (x[i] > 0) << i;
                code[i] = codes[min(cofs[i] + max(x[i] - 1, 0), total - 1)];  // at x_i = 0 unused, but a code
            }
            int pair[NP];
            {
                int p = 0;
#pragma unroll
                for (int i = 0; i < K; ++i)
#pragma unroll
                    for (int j = i + 1; j < K; ++j) pair[p++] = sub[code[i] * A + code[j]] - 2 * gap;
            }
            int first = 0, spfirst = 0;
            unsigned mine[NW];
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const int m = 32 * w + lane;
                const bool ok = m > 0 && m < NM && (m & ~open) == 0;
                int sp = u * __popc(m);  // gap terms: u per residue, less 2 gap per pair of residues
                int p = 0;
                int64_t g = 0;
#pragma unroll
                for (int i = 0; i < K; ++i) {
                    const int bi = (m >> i) & 1;
                    g += off[at[i] + x[i] - (ok ? bi : 0)];
#pragma unroll
                    for (int j = i + 1; j < K; ++j, ++p)
                        if (bi & (m >> j)) sp += pair[p];
                }
                bool hit = false;
                if (ok) {
                    const int h = ((Q[g] - (W - m)) >> K) + u * (S - __popc(m));
                    hit = h + sp + acc >= thr;
                }
                mine[w] = __ballot_sync(kFull, hit);
                if (!first && mine[w]) {  // uniform
                    const int l = __ffs(mine[w]) - 1;
                    first = 32 * w + l;
                    spfirst = __shfl_sync(kFull, sp, l);
                    mine[w] &= mine[w] - 1;
                }
            }
            if (first) {  // follow the lowest mask, the others stay on the stack
                if (lane == 0) {
#pragma unroll
                    for (int w = 0; w < NW; ++w) hits[(size_t)d * NW + w] = mine[w];
                    accs[d] = acc;
                    path[d] = (uint8_t)first;
                }
#pragma unroll
                for (int i = 0; i < K; ++i) x[i] -= (first >> i) & 1;
                S -= __popc(first);
                W -= first;
                acc += spfirst;
                ++d;
                continue;
            }
        }
        // back to the deepest depth with a mask left, 32 depths at a time
        __syncwarp();
        int found = -1;
        while (d > 0 && found < 0) {
            const int j = d - 1 - lane;
            unsigned any = 0;
            int pm = 0;
            if (j >= 0) {
#pragma unroll
                for (int w = 0; w < NW; ++w) any |= hits[(size_t)j * NW + w];
                pm = path[j];
            }
            const unsigned has = __ballot_sync(kFull, any != 0);
            const int n = has ? __ffs(has) : min(d, 32);  // depths to undo
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const unsigned moved = __ballot_sync(kFull, (pm >> i) & 1) & (n == 32 ? kFull : (1u << n) - 1);
                x[i] += __popc(moved);
                S += __popc(moved);
                W += __popc(moved) << i;
            }
            d -= n;
            if (has) found = d;
        }
        if (found < 0) break;  // nothing left
        if (count == max_count) {
            more = 1;
            break;
        }
        // its lowest mask left: the column's score from its residues
        int m = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const unsigned h = hits[(size_t)d * NW + w];
            if (!m && h) {
                m = 32 * w + __ffs(h) - 1;
                __syncwarp();
                if (lane == 0) hits[(size_t)d * NW + w] = h & (h - 1);
            }
        }
        acc = accs[d] + u * __popc(m);
#pragma unroll
        for (int i = 0; i < K; ++i)
#pragma unroll
            for (int j = i + 1; j < K; ++j)
                if ((m >> i) & (m >> j) & 1)
                    acc += sub[codes[cofs[i] + x[i] - 1] * A + codes[cofs[j] + x[j] - 1]] - 2 * gap;
        __syncwarp();
        if (lane == 0) path[d] = (uint8_t)m;
#pragma unroll
        for (int i = 0; i < K; ++i) x[i] -= (m >> i) & 1;
        S -= __popc(m);
        W -= m;
        ++d;
    }
    if (lane == 0) {
        o.count_more[0] = count;
        o.count_more[1] = more;
    }
}

template <int K>
cudaError_t launch_near(const ProblemDesc *d_prob, IODesc io, int64_t delta, int32_t max_count, NearOut o, size_t bytes,
                        cudaStream_t s) {
    const int in_smem = bytes <= (size_t)kNearSmem;
    cudaError_t e = cudaFuncSetAttribute(near_optimal_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, kNearSmem);
    if (e != cudaSuccess) return e;
    near_optimal_kernel<K><<<1, kNearThreads, in_smem ? bytes : 0, s>>>(d_prob, io, delta, max_count, o, in_smem);
    return cudaGetLastError();
}

}  // namespace

size_t near_optimal_work_bytes(int k, int64_t len_sum) {
    const size_t b = near_bytes(k, len_sum);
    return b <= (size_t)kNearSmem ? 0 : b;
}

cudaError_t launch_near_optimal(int k, int64_t len_sum, const ProblemDesc *d_prob, IODesc io, int64_t delta,
                                int32_t max_count, NearOut o, cudaStream_t s) {
    const size_t bytes = near_bytes(k, len_sum);
    switch (k) {
        case 2: return launch_near<2>(d_prob, io, delta, max_count, o, bytes, s);
        case 3: return launch_near<3>(d_prob, io, delta, max_count, o, bytes, s);
        case 4: return launch_near<4>(d_prob, io, delta, max_count, o, bytes, s);
        case 5: return launch_near<5>(d_prob, io, delta, max_count, o, bytes, s);
        case 6: return launch_near<6>(d_prob, io, delta, max_count, o, bytes, s);
        case 7: return launch_near<7>(d_prob, io, delta, max_count, o, bytes, s);
        case 8: return launch_near<8>(d_prob, io, delta, max_count, o, bytes, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace msadp
