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
// The fill is the column or band kernel in the form that keeps every cell's score, or
// the generic tile kernel, which keeps the packed key of every cell:
// Q(x) = H'(x) 2^k + W(x) with H'(x) = H(x) - gap (k - 1) |x|_1 and
// W(x) = sum_i 2^i x_i, so H(x) = (Q(x) - W(x)) / 2^k + gap (k - 1) |x|_1
// exactly (and in 32 bits: every sum compared below is the score of an alignment,
// which the encode step's range check keeps in range). The other two keep
// H'(x) 2^k plus a tag below 2^k, so there W is left out.
//
// In the depth-first form one warp walks, and what bounds it is the chain of one node: residue codes and
// offsets from shared memory, one score per lane, a ballot. At a node every mask is
// judged at once, a lane per mask (and 32 masks per round), and the set that
// qualifies goes on the stack, so going back costs no judging: the lanes look 32
// depths at a time for the deepest one with a mask left and count the moves to undo
// with one ballot per axis. The offset of a cell is a sum of one term per axis in
// every layout of the scores, so the terms are tabulated per coordinate once.
// 256 alignments within 3 of the optimum of a related 120 x 110 x 130 triple: 37.9 ms when
// the walk went back one column at a time, judging again, with positions in local memory;
// 3.58 ms depth first now, 0.32 level by level (near_beam_kernel, the form for shorter
// sequences, which this problem takes).
#include "device_common.cuh"

#include <algorithm>

namespace msadp {

namespace {

constexpr int kNearThreads = 256;
constexpr int kNearSmem = 160 * 1024;  // tables and stack beyond this stay in global memory

// Term of coordinate v of axis i in the element offset of a cell's score: row-major
// (qstride) for k <= 3, tile-major (the traceback's layout 2) for k >= 4; the layouts of
// the kernels that keep scores.
__device__ __forceinline__ int64_t axis_offset(const ProblemDesc &P, int i, int v) {
    if (P.kept) return P.k == 2 ? band2_kept_term(i, v, P.rho[1]) : c3::kept_term(i, v, P.G[1], P.rho[2]);
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
    const int32_t *Q = P.kept ? P.kept : P.Q;
    const int withw = P.kept ? 0 : -1;  // the scores' W part
    const int opt = ((Q[corner] - (W & withw)) >> K) + u * S;
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
                    const int h = ((Q[g] - ((W - m) & withw)) >> K) + u * (S - __popc(m));
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

// The same enumeration level by level: every partial alignment that qualifies leads to
// at least one alignment, so of the partial alignments of d columns, in order, only the
// first max_count can be the start of one of the first max_count alignments. They are
// kept as slots in shared memory; at each level a group of 2^k lanes per slot judges
// its masks, and a count over the ballots lays the children down in order (a slot that
// has reached the origin is carried on as it is). A level is one chain of loads, a
// ballot and a barrier, as a node of the depth-first walk is, but takes all slots: 256
// alignments of another such triple, 143 levels: 0.263 against 3.62 ms node by node. A level
// costs more than a node, though, and the walk judges only the cells of the alignments
// it stores, which on long sequences differ in their last few columns. So up to
// kBeamLength residues this way (300 x 300, 30 alignments: 0.187 against 0.376 ms;
// 120 x 110 x 130, all 660 of up to 2,000: 0.485 against 9.96) and the walk beyond (800 x
// 700 unrelated, 90: 0.621 against 0.455 ms; 5000 x 4800, 512: 12.2 against 7.64), and
// beyond kBeamRounds rounds of a CTA's lanes per level.
//
// A slot carries its last up to 8 masks packed in a word and its ancestor's slot at the
// level the word began; every 8 levels the two go to the history, from which each
// alignment's columns are read back at the end, 8 at a time.
constexpr int kBeamThreads = 1024, kBeamRounds = 16, kBeamLength = 1024;
__host__ __device__ constexpr int beam_group(int K) { return K < 5 ? 1 << K : 32; }  // lanes judging a slot
__host__ __device__ constexpr int beam_slots(int K) { return kBeamThreads / beam_group(K); }  // slots a round takes
__host__ __device__ constexpr int beam_words(int K) { return (K + 4) | 1; }  // position, score, ancestor, two words of masks (odd: no bank conflicts)
__host__ __device__ constexpr size_t beam_history_rows(int64_t len_sum) { return (size_t)len_sum / 8 + 1; }
size_t beam_tables(int k, int64_t len_sum) { return ((size_t)len_sum + k) * 8 + (((size_t)len_sum + 15) & ~(size_t)15) + 16; }
size_t beam_state(int k, int32_t max_count) { return (size_t)2 * beam_words(k) * max_count * 4; }
bool beam_fits(int k, int64_t len_sum, int32_t max_count) {
    return max_count <= kBeamRounds * beam_slots(k) && len_sum <= kBeamLength &&
           beam_tables(k, len_sum) + beam_state(k, max_count) <= (size_t)kNearSmem;
}

template <int K>
__global__ void __launch_bounds__(kBeamThreads) near_beam_kernel(const ProblemDesc *probs, IODesc io, int64_t delta,
                                                                 int32_t max_count, NearOut o) {
    constexpr int NW = near_words(K), NM = 1 << K, NP = K * (K - 1) / 2;
    constexpr int GW = beam_group(K), SPW = 32 / GW, NS = beam_words(K);
    extern __shared__ __align__(16) unsigned char near_smem[];
    __shared__ int sub[MSA_MAX_ALPHABET * MSA_MAX_ALPHABET];
    __shared__ int counts[2][32];
    __shared__ int dead;  // a slot away from the origin that no move leads on from
    const ProblemDesc &P = probs[0];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int nthreads = blockDim.x, nwarps = nthreads / 32;
    const int A = P.A, total = P.len_sum;
    if (ld_volatile(&P.istat->status) != 0) {  // the fill did not complete: nothing to enumerate
        if (tid < 2) o.count_more[tid] = 0;
        return;
    }
    int64_t *off = reinterpret_cast<int64_t *>(near_smem);
    int *state = reinterpret_cast<int *>(off + total + K);
    uint8_t *codes = reinterpret_cast<uint8_t *>(state + 2 * (size_t)NS * max_count);
    int cofs[K], at[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        cofs[i] = P.cofs[i];
        at[i] = cofs[i] + i;
        for (int v = tid; v < P.rho[i]; v += nthreads) off[at[i] + v] = axis_offset(P, i, v);
    }
    for (int c = tid; c < total; c += nthreads) codes[c] = P.codes[c];
    for (int c = tid; c < A * A; c += nthreads) sub[c] = io.subst[c];
    if (tid < 64) counts[tid >> 5][lane] = 0;
    auto slot_words = [&](int buf, int slot) { return state + (buf * max_count + slot) * NS; };
    if (tid == 0) {
        dead = 0;
        for (int w = 0; w < NS; ++w) state[w] = w < K ? P.len[w] : 0;
    }
    __syncthreads();

    if (max_count <= SPW) {  // one warp takes every level
        if (warp > 0) return;
        nthreads = 32, nwarps = 1;
    }
    const int gap = io.gap, u = gap * (K - 1);
    const int32_t *Q = P.kept ? P.kept : P.Q;
    const int withw = P.kept ? 0 : -1;  // the scores' W part
    int thr;
    {
        int S = 0, W = 0;
        int64_t corner = 0;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            S += P.len[i];
            W += P.len[i] << i;
            corner += off[at[i] + P.len[i]];
        }
        const int opt = ((Q[corner] - (W & withw)) >> K) + u * S;
        thr = delta > (int64_t)opt - INT32_MIN ? INT32_MIN : (int)(opt - delta);
    }
    uint64_t *hwords = reinterpret_cast<uint64_t *>(o.work);
    int32_t *hprev = reinterpret_cast<int32_t *>(hwords + beam_history_rows(total) * max_count);
    int n = 1, level = 0, more_left = 0, cur = 0, cb = 0;
    // (every level but the last lowers the sum of every unfinished slot's coordinates)
    while (level <= total) {
        int base = 0, live = 0, more = 0;
        const bool flush = (level & 7) == 7;
        for (int s0 = 0; s0 < n && !more; s0 += nwarps * SPW) {
            const int first = s0 + warp * SPW, slot = first + lane / GW;
            unsigned mine[NW];
            int sps[NW];
            int x[K], acc = 0, S = 0, cnt = 0;
#pragma unroll
            for (int w = 0; w < NW; ++w) mine[w] = 0;
            if (first < n) {
                const int *st = slot_words(cur, min(slot, n - 1));
                int W = 0, open = 0, code[K];
#pragma unroll
                for (int i = 0; i < K; ++i) {
                    x[i] = st[i];
                    S += x[i];
                    W += x[i] << i;
                    open |= (x[i] > 0) << i;
                    code[i] = x[i] > 0 ? codes[cofs[i] + x[i] - 1] : 0;  // (no residue to read where all are empty)
                }
                acc = st[K];
                int pair[NP];
                {
                    int p = 0;
#pragma unroll
                    for (int i = 0; i < K; ++i)
#pragma unroll
                        for (int j = i + 1; j < K; ++j) pair[p++] = sub[code[i] * A + code[j]] - 2 * gap;
                }
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    const int m = 32 * w + lane % GW;
                    const bool ok = slot < n && m > 0 && m < NM && (m & ~open) == 0;
                    int sp = u * __popc(m);
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
                    sps[w] = sp;
                    bool hit = false;
                    if (ok) {
                        const int h = ((Q[g] - ((W - m) & withw)) >> K) + u * (S - __popc(m));
                        hit = h + sp + acc >= thr;
                        live |= hit;
                    } else if (m == 0 && slot < n) {
                        hit = S == 0;  // finished: carried on
                    }
                    mine[w] = __ballot_sync(kFull, hit);
                    cnt += __popc(mine[w]);
                }
                unsigned any = 0;
#pragma unroll
                for (int w = 0; w < NW; ++w) any |= mine[w] >> (lane & ~(GW - 1));
                if (slot < n && (any & (GW == 32 ? kFull : (1u << GW % 32) - 1)) == 0) dead = 1;
            }
            if (lane == 0) counts[cb][warp] = cnt;
            __syncthreads();
            const int c = counts[cb][lane];
            int idx = base + (int)__reduce_add_sync(kFull, (unsigned)(lane < warp ? c : 0));
            base += (int)__reduce_add_sync(kFull, (unsigned)c);
            cb ^= 1;
            more = base > max_count || (base == max_count && s0 + nwarps * SPW < n);
            if (cnt == 0) continue;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const int i0 = idx + __popc(mine[w] & ((1u << lane) - 1));
                idx += __popc(mine[w]);
                if (!((mine[w] >> lane) & 1) || i0 >= max_count) continue;
                const int m = 32 * w + lane % GW;
                const int *st = slot_words(cur, slot);
                int *child = slot_words(cur ^ 1, i0);
#pragma unroll
                for (int i = 0; i < K; ++i) child[i] = x[i] - ((m >> i) & 1);
                child[K] = acc + (m ? sps[w] : 0);
                uint2 packed = make_uint2((unsigned)st[K + 2], (unsigned)st[K + 3]);
                const unsigned put = (unsigned)m << 8 * (level & 3);
                if (level & 4)
                    packed.y |= put;
                else
                    packed.x |= put;
                int from = st[K + 1];
                if (flush) {
                    const size_t h = (size_t)(level >> 3) * max_count + i0;
                    hwords[h] = (uint64_t)packed.y << 32 | packed.x;
                    hprev[h] = from;
                    packed = make_uint2(0, 0);
                    from = i0;
                }
                child[K + 1] = from;
                child[K + 2] = (int)packed.x;
                child[K + 3] = (int)packed.y;
            }
        }
        n = min(base, max_count);
        cur ^= 1;
        ++level;
        more_left |= more;
        if (!__syncthreads_or(live)) break;
    }
    // every slot stands at the origin: its columns, first (the last move) to last
    for (int slot = tid; slot < n; slot += nthreads) {
        uint8_t *dst = o.masks + (int64_t)slot * total;
        const int *st = slot_words(cur, slot);
        uint64_t w = (uint64_t)(unsigned)st[K + 3] << 32 | (unsigned)st[K + 2];
        int from = st[K + 1], c = 0;
        for (int row = (level >> 3) - 1;; --row) {
            for (; w; w <<= 8)
                if (w >> 56) dst[c++] = (uint8_t)(w >> 56);
            if (row < 0) break;
            const size_t h = (size_t)row * max_count + from;
            w = hwords[h];
            from = hprev[h];
        }
        o.ncols[slot] = c;
        o.scores[slot] = st[K];
    }
    if (tid == 0) {
        o.count_more[0] = n;
        o.count_more[1] = dead ? 2 : more_left;  // 2: an inconsistent tensor
    }
}

template <int K>
cudaError_t launch_beam(const ProblemDesc *d_prob, IODesc io, int64_t delta, int64_t len_sum, int32_t max_count, NearOut o,
                        cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(near_beam_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, kNearSmem);
    if (e != cudaSuccess) return e;
    // as many warps as a level may fill (eight at least, for the tables and the columns)
    const int warps = std::min(kBeamThreads / 32, std::max(8, (max_count * beam_group(K) + 31) / 32));
    near_beam_kernel<K><<<1, 32 * warps, beam_tables(K, len_sum) + beam_state(K, max_count), s>>>(d_prob, io, delta,
                                                                                                 max_count, o);
    return cudaGetLastError();
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

size_t near_optimal_work_bytes(int k, int64_t len_sum, int32_t max_count) {
    if (beam_fits(k, len_sum, max_count)) return beam_history_rows(len_sum) * max_count * 12;
    const size_t b = near_bytes(k, len_sum);
    return b <= (size_t)kNearSmem ? 0 : b;
}

cudaError_t launch_near_optimal(int k, int64_t len_sum, const ProblemDesc *d_prob, IODesc io, int64_t delta,
                                int32_t max_count, NearOut o, cudaStream_t s) {
    const size_t bytes = near_bytes(k, len_sum);
    if (beam_fits(k, len_sum, max_count)) switch (k) {
            case 2: return launch_beam<2>(d_prob, io, delta, len_sum, max_count, o, s);
            case 3: return launch_beam<3>(d_prob, io, delta, len_sum, max_count, o, s);
            case 4: return launch_beam<4>(d_prob, io, delta, len_sum, max_count, o, s);
            case 5: return launch_beam<5>(d_prob, io, delta, len_sum, max_count, o, s);
            case 6: return launch_beam<6>(d_prob, io, delta, len_sum, max_count, o, s);
            case 7: return launch_beam<7>(d_prob, io, delta, len_sum, max_count, o, s);
            case 8: return launch_beam<8>(d_prob, io, delta, len_sum, max_count, o, s);
        }
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
