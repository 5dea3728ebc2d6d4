// Top-K softmax over per-position next-token logits.  Selection is exact (logit descending, index
// ascending, -0 = +0).
//
// K <= 128, and calls that ask for no selected set (only lse / log2 P): topk_stream_kernel, which reads
// a row once, any alignment (see there); topk_pipe_kernel where the rows are long and many.  K > 128: topk_softmax_kernel, one block a row: thread maxima bound
// the K-th logit where K allows it; else a 4096-bin histogram of the order-preserving 16-bit key finds the
// bin that holds the K-th largest, a 16-way refinement finds the key itself, and equal keys are taken in
// index order.
// Reductions use warp shuffles in a fixed order, so results are bit-reproducible from run to run.
#include <algorithm>
#include <type_traits>

#include "plc_common.cuh"

namespace plc {
namespace {

constexpr int kBins = 4096;
constexpr int kCandCap = 1024;

__device__ __forceinline__ uint32_t key_of(uint32_t u) {
    u &= 0xffffu;
    if ((u & 0x7fffu) == 0) u = 0;                  // -0 and +0 are the same logit
    return (u & 0x8000u) ? (~u & 0xffffu) : (u | 0x8000u);
}
__device__ __forceinline__ uint32_t bits_of_key(uint32_t key) {
    return (key & 0x8000u) ? (key & 0x7fffu) : (~key & 0xffffu);
}
__device__ __forceinline__ float val_of_key(uint32_t key) {
    return __half2float(__ushort_as_half((unsigned short)bits_of_key(key)));
}
constexpr uint32_t kKeyNegInf = 0x03ffu;            // key_of(0xfc00)

template <int THREADS>
struct __align__(16) Smem {
    uint32_t hist[kBins];
    uint32_t sub[16];
    uint32_t sel_key[kCandCap];
    int32_t sel_idx[kCandCap];
    uint32_t cand_key[kCandCap];
    int32_t cand_idx[kCandCap];
    float ek[kCandCap];
    uint32_t red_k[THREADS / 32], red_t[THREADS / 32];
    float red_s[THREADS / 32];
    int scan[THREADS / 32];
    int nsel, ncand, bstar, count_above, cstar, thr, need, neq, running, nlist, nhit;
    float sum_k;
};

// Exclusive scan of one int per thread over the block (thread order); total to all threads.
template <int THREADS>
__device__ __forceinline__ int block_excl_scan(int v, int* scratch, int& total) {
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += t;
    }
    __syncthreads();                                 // scratch free
    if (lane == 31) scratch[wid] = inc;
    __syncthreads();
    int base = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) {
        int x = scratch[w];
        if (w < wid) base += x;
        tot += x;
    }
    total = tot;
    return base + inc - v;
}

// Calls f(index, raw binary16 bits) for the elements of the row that this thread owns in tile `t`.
// A tile is THREADS*8 consecutive elements; a thread owns 8 consecutive ones.
template <bool VEC, int THREADS, class F>
__device__ __forceinline__ void for_tile(const __half* row, int V, int t, F&& f) {
    int i0 = t * (THREADS * 8) + threadIdx.x * 8;
    if (VEC) {
        if (i0 < V) {                                // V % 8 == 0: the 8 are all in range
            uint4 r = *reinterpret_cast<const uint4*>(row + i0);
            uint32_t wds[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                f(i0 + 2 * j, wds[j] & 0xffffu);
                f(i0 + 2 * j + 1, wds[j] >> 16);
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (i0 + j < V) f(i0 + j, (uint32_t)__half_as_ushort(row[i0 + j]));
    }
}

// exp(x - l_max) as 2^(x log2(e) - l_max log2(e)): one fused multiply-add and one ex2.approx (relative
// error about 2e-6 at the arguments that matter, inside the tolerance of lse and Z_k; results below
// 2^-126 flush to zero).  nb = -l_max log2(e).
__device__ __forceinline__ float exp_rel(float x, float nb) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__fmaf_rn(x, 1.44269504088896341f, nb)));
    return r;
}

__device__ __forceinline__ uint32_t hmax2_bits(uint32_t a, uint32_t b) {
    __half2 r = __hmax2(*reinterpret_cast<__half2*>(&a), *reinterpret_cast<__half2*>(&b));
    return *reinterpret_cast<uint32_t*>(&r);
}

// Sorts n_pad (a power of two) order words in shared memory, largest first, with the block.
template <int THREADS, class W>
__device__ __forceinline__ void bitonic_desc(W* v, int n_pad) {
    for (int k = 2; k <= n_pad; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = threadIdx.x; t < (n_pad >> 1); t += THREADS) {
                const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1));       // lower index of the pair
                const W a = v[i], b = v[i | j];
                const bool desc = (i & k) == 0;
                if ((a < b) == desc) { v[i] = b; v[i | j] = a; }
            }
            __syncthreads();
        }
}

// Radix select of the K largest keys of the row into sm.sel_* (unordered); three or more passes
// over the row.
template <bool VEC, int THREADS>
__device__ void select_by_histogram(Smem<THREADS>& sm, const __half* row, int V, int K, int ntiles) {
    const int tid = threadIdx.x;
    for (int i = tid; i < kBins; i += THREADS) sm.hist[i] = 0;
    if (tid < 16) sm.sub[tid] = 0;
    if (tid == 0) { sm.nsel = 0; sm.ncand = 0; sm.running = 0; }
    __syncthreads();
    // Pass A: histogram of the top 12 key bits (keys order like the logits).
    for (int t = 0; t < ntiles; ++t)
        for_tile<VEC, THREADS>(row, V, t, [&](int, uint32_t bits) { atomicAdd(&sm.hist[key_of(bits) >> 4], 1u); });
    __syncthreads();
    // Bin that holds the K-th largest key: thread t owns BPT bins going down from 4095 - BPT*t.
    {
        constexpr int BPT = kBins / THREADS;
        int local = 0;
#pragma unroll
        for (int j = 0; j < BPT; ++j) local += (int)sm.hist[kBins - 1 - (tid * BPT + j)];
        int total;
        int excl = block_excl_scan<THREADS>(local, sm.scan, total);
        if (excl < K && K <= excl + local) {
            int cum = excl;
            for (int j = 0; j < BPT; ++j) {
                int b = kBins - 1 - (tid * BPT + j);
                int c = (int)sm.hist[b];
                if (cum + c >= K) { sm.bstar = b; sm.count_above = cum; sm.cstar = c; break; }
                cum += c;
            }
        }
    }
    __syncthreads();
    const int bstar = sm.bstar, cstar = sm.cstar, count_above = sm.count_above;
    const bool use_cand = cstar <= kCandCap;
    // Pass B: everything above the bin is selected; inside the bin refine on the low 4 key bits.
    for (int t = 0; t < ntiles; ++t)
        for_tile<VEC, THREADS>(row, V, t, [&](int i, uint32_t bits) {
            uint32_t key = key_of(bits);
            int bin = (int)(key >> 4);
            if (bin > bstar) {
                int slot = atomicAdd(&sm.nsel, 1);
                sm.sel_key[slot] = key; sm.sel_idx[slot] = i;
            } else if (bin == bstar) {
                atomicAdd(&sm.sub[key & 15u], 1u);
                if (use_cand) {
                    int slot = atomicAdd(&sm.ncand, 1);
                    sm.cand_key[slot] = key; sm.cand_idx[slot] = i;
                }
            }
        });
    __syncthreads();
    if (tid == 0) {
        int need1 = K - count_above, cum = 0;
        for (int j = 15; j >= 0; --j) {
            int c = (int)sm.sub[j];
            if (cum + c >= need1) { sm.thr = (bstar << 4) | j; sm.need = need1 - cum; sm.neq = c; break; }
            cum += c;
        }
    }
    __syncthreads();
    const uint32_t thr = (uint32_t)sm.thr;
    const int need = sm.need, neq = sm.neq;
    if (use_cand) {
        const int nc = sm.ncand;
        for (int c = tid; c < nc; c += THREADS) {
            uint32_t key = sm.cand_key[c];
            int idx = sm.cand_idx[c];
            bool take = key > thr;
            if (key == thr) {
                if (need == neq) take = true;
                else {
                    int rank = 0;
                    for (int j = 0; j < nc; ++j) rank += (sm.cand_key[j] == thr && sm.cand_idx[j] < idx);
                    take = rank < need;
                }
            }
            if (take) {
                int slot = atomicAdd(&sm.nsel, 1);
                sm.sel_key[slot] = key; sm.sel_idx[slot] = idx;
            }
        }
    } else {
        // Pass C (large tie groups): re-read the row; equal keys are taken in index order.
        for (int t = 0; t < ntiles; ++t) {
            int cnt = 0;
            for_tile<VEC, THREADS>(row, V, t, [&](int i, uint32_t bits) {
                uint32_t key = key_of(bits);
                if ((int)(key >> 4) == bstar && key > thr) {
                    int slot = atomicAdd(&sm.nsel, 1);
                    sm.sel_key[slot] = key; sm.sel_idx[slot] = i;
                }
                cnt += (key == thr);
            });
            int total;
            int rank = block_excl_scan<THREADS>(cnt, sm.scan, total) + sm.running;
            for_tile<VEC, THREADS>(row, V, t, [&](int i, uint32_t bits) {
                uint32_t key = key_of(bits);
                if (key == thr) {
                    if (rank < need) {
                        int slot = atomicAdd(&sm.nsel, 1);
                        sm.sel_key[slot] = key; sm.sel_idx[slot] = i;
                    }
                    ++rank;
                }
            });
            __syncthreads();
            if (tid == 0) sm.running += total;
            __syncthreads();
        }
    }
    __syncthreads();
    // Order the K selected by (key descending, index ascending): a sort of packed order words in the
    // histogram's memory.
    unsigned long long* w = reinterpret_cast<unsigned long long*>(sm.hist);
    int n_pad = 256;
    while (n_pad < K) n_pad <<= 1;
    for (int k = tid; k < n_pad; k += THREADS)
        w[k] = k < K ? ((unsigned long long)sm.sel_key[k] << 32) | (0xffffffffu - (uint32_t)sm.sel_idx[k]) : 0ull;
    __syncthreads();
    bitonic_desc<THREADS>(w, n_pad);
    for (int k = tid; k < K; k += THREADS) {
        sm.cand_key[k] = (uint32_t)(w[k] >> 32); sm.cand_idx[k] = (int)(0xffffffffu - (uint32_t)w[k]);
    }
    __syncthreads();
}

// Entry k of a row's pairs: byte offset of the candidate's table row (its index where a table's rows span
// 4 GB or more) and weight, in the order in which the gather's lanes read them: the entries of one of
// the 1 << pair_rows row groups of a warp-wide load follow each other.
__device__ __forceinline__ void put_pair(const TopkArgs& a, long long rowi, int k, int idx, float w) {
    const int at = (k & ((1 << a.pair_rows) - 1)) * (a.Kp >> a.pair_rows) + (k >> a.pair_rows);
    a.pairs[rowi * a.Kp + at] = make_int2((int)((unsigned)idx * (unsigned)a.pair_mul), __float_as_int(w));
}

// log2 P of the row's token and, for the adaptive step (Def. 7), b = max(1, floor(b0 h / hbar)) capped at
// b0 + extra, decided in binary32.
__device__ __forceinline__ void put_surprisal(const TopkArgs& a, long long rowi, const __half* row, float lse) {
    const int tk = a.tokens[rowi];
    const float v = (tk >= 0 && tk < a.V) ? (__half2float(row[tk]) - lse) * 1.44269504088896341f : __int_as_float(0x7fc00000);
    if (a.logp2) a.logp2[rowi] = v;
    if (a.step_exp || a.bits_out) {
        const float r = __fmul_rn((float)a.b0, __fdiv_rn(-v, a.hbar));
        int b = (r >= 1.0f) ? (int)floorf(r) : 1;
        b = min(b, a.b0 + a.extra);
        if (a.step_exp) a.step_exp[rowi] = a.b0 - b;
        if (a.bits_out) a.bits_out[rowi] = b;
    }
}

// What a row gives beside its selection.
__device__ __forceinline__ void put_row(const TopkArgs& a, long long rowi, const __half* row, float lse) {
    if (a.lse) a.lse[rowi] = lse;
    if (a.tokens && (a.logp2 || a.step_exp || a.bits_out)) put_surprisal(a, rowi, row, lse);
}

__device__ __forceinline__ void zero_tickets(const TopkArgs& a) {
    if (a.tickets && blockIdx.x == 0)
        for (int i = threadIdx.x; i < kTicketWords; i += blockDim.x) a.tickets[i] = 0u;
}

// K > 128: a block a row, two passes over it.  The first takes a maximum per thread.  Where a warp's share of K
// is at most half of its lanes (K <= 256 with 16 warps: rows of more than 65536 logits) the per_warp-th largest
// of a warp's maxima, the smallest over the warps, bounds the K-th logit from below; the second pass, the
// sum, then notes the groups of 8 that reach it, and their logits, a few more than K, are sorted.
// Otherwise, and where ties overflow the list, select_by_histogram reads the row again.
// (4096 rows of 128256, K = 256: 1294 us by histograms, 510 so; K = 1024, 1024 rows: maxima key by key 425, packed
// 370.)
template <bool VEC, int THREADS>
__global__ void __launch_bounds__(THREADS) topk_softmax_kernel(TopkArgs a) {
    constexpr int NW = THREADS / 32;
    __shared__ Smem<THREADS> sm;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int V = a.V, K = a.K;
    const int ntiles = (V + THREADS * 8 - 1) / (THREADS * 8);
    const int per_warp = (K + NW - 1) / NW;
    const bool bounded = THREADS == 512 && per_warp <= 16;              // K <= 256
    unsigned long long* list = reinterpret_cast<unsigned long long*>(sm.hist);           // idle until the histograms
    static_assert(kCandCap * sizeof(unsigned long long) <= sizeof(sm.hist), "the list lives there");
    chain_next();
    chain_wait();
    zero_tickets(a);
    for (long long rowi = blockIdx.x; rowi < a.N; rowi += gridDim.x) {
        if (a.pos_begin || a.pos_end) {
            int s = (int)(rowi / a.n_per_session), i = (int)(rowi % a.n_per_session);
            int b = a.pos_begin ? a.pos_begin[s] : 0, e = a.pos_end ? a.pos_end[s] : a.n_per_session;
            if (i < b || i >= e) continue;
        }
        const __half* row = a.logits + rowi * (long long)V;
        if (tid == 0) { sm.nlist = 0; sm.nhit = 0; }
        // Pass 0 (HBM): the maximum.
        uint32_t m2 = 0xfc00fc00u;                                   // (-inf, -inf); NaN loses every maximum
        if (VEC) {
#pragma unroll 4
            for (int t = 0; t < ntiles; ++t) {
                const int i0 = t * (THREADS * 8) + tid * 8;
                if (i0 < V) {
                    const uint4 r = *reinterpret_cast<const uint4*>(row + i0);
                    m2 = hmax2_bits(m2, hmax2_bits(hmax2_bits(r.x, r.y), hmax2_bits(r.z, r.w)));
                }
            }
        } else {
            for (int t = 0; t < ntiles; ++t)
                for_tile<VEC, THREADS>(row, V, t, [&](int, uint32_t bits) { m2 = hmax2_bits(m2, bits * 0x10001u); });
        }
        const uint32_t tkey = tid * 8 < V ? max(key_of(m2 & 0xffffu), key_of(m2 >> 16)) : 0u;
        const uint32_t wmax = __reduce_max_sync(kFull, tkey);
        uint32_t wth = 0;
        if (bounded) {
            uint32_t v = tkey;
            for (int r = 0; r < per_warp; ++r) {
                wth = __reduce_max_sync(kFull, v);
                const uint32_t eq = __ballot_sync(kFull, v == wth);
                if (lane == __ffs(eq) - 1) v = 0;
            }
        }
        if (lane == 0) { sm.red_k[wid] = wmax; sm.red_t[wid] = wth; }
        __syncthreads();
        uint32_t km = sm.red_k[0], theta = sm.red_t[0];
#pragma unroll
        for (int w = 1; w < NW; ++w) { km = max(km, sm.red_k[w]); theta = min(theta, sm.red_t[w]); }
        theta = max(theta, kKeyNegInf);
        const float lmax = val_of_key(max(km, kKeyNegInf));
        // Pass 1 (L2): sum of exp(l - l_max), and what reaches the bound.
        const float nb = -lmax * 1.44269504088896341f;
        const uint32_t th2 = bits_of_key(theta) * 0x10001u;
        float s = 0.f;
        if (VEC) {
#pragma unroll 2
            for (int t = 0; t < ntiles; ++t) {
                const int i0 = t * (THREADS * 8) + tid * 8;
                if (i0 < V) {
                    const uint4 r = *reinterpret_cast<const uint4*>(row + i0);
                    const uint32_t wds[4] = {r.x, r.y, r.z, r.w};
                    const uint32_t top = hmax2_bits(hmax2_bits(r.x, r.y), hmax2_bits(r.z, r.w));
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&wds[j]));
                        s += exp_rel(f.x, nb);
                        s += exp_rel(f.y, nb);
                    }
                    // a group is only noted here (few lanes get here); the noted ones are taken apart after the pass
                    if (bounded && __hge2_mask(*reinterpret_cast<const __half2*>(&top), *reinterpret_cast<const __half2*>(&th2))) {
                        const int slot = atomicAdd(&sm.nhit, 1);
                        if (slot < kCandCap) sm.sel_idx[slot] = i0;              // sel_idx is idle until the histograms
                    }
                }
            }
        } else {
            for (int t = 0; t < ntiles; ++t)
                for_tile<VEC, THREADS>(row, V, t, [&](int i, uint32_t bits) {
                    s += exp_rel(__half2float(__ushort_as_half((unsigned short)bits)), nb);
                    const uint32_t key = key_of(bits);
                    if (bounded && key >= theta) {
                        const int slot = atomicAdd(&sm.nlist, 1);
                        if (slot < kCandCap) list[slot] = ((unsigned long long)key << 32) | (0xffffffffu - (uint32_t)i);
                    }
                });
        }
        s = warp_sum(s);
        if (lane == 0) sm.red_s[wid] = s;
        __syncthreads();
        float sum_all = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) sum_all += sm.red_s[w];
        if (VEC && bounded) {
            const int nhit = sm.nhit;
            for (int t = tid; t < min(nhit, kCandCap); t += THREADS) {
                const int i0 = sm.sel_idx[t];
                const uint4 r = *reinterpret_cast<const uint4*>(row + i0);
                const uint32_t wds[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t ge = __hge2_mask(*reinterpret_cast<const __half2*>(&wds[j]), *reinterpret_cast<const __half2*>(&th2));
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if ((ge >> (16 * h)) & 1u) {
                            const int slot = atomicAdd(&sm.nlist, 1);
                            if (slot < kCandCap) list[slot] = ((unsigned long long)key_of(wds[j] >> (16 * h)) << 32) | (0xffffffffu - (uint32_t)(i0 + 2 * j + h));
                        }
                }
            }
            if (tid == 0 && nhit > kCandCap) atomicAdd(&sm.nlist, kCandCap + 1);       // too many
            __syncthreads();
        }
        const int nlist = sm.nlist;
        if (bounded && nlist >= K && nlist <= kCandCap) {
            int n_pad = 256;
            while (n_pad < nlist) n_pad <<= 1;
            for (int k = nlist + tid; k < n_pad; k += THREADS) list[k] = 0;              // orders after everything
            __syncthreads();
            bitonic_desc<THREADS>(list, n_pad);
            for (int k = tid; k < K; k += THREADS) {
                sm.cand_key[k] = (uint32_t)(list[k] >> 32); sm.cand_idx[k] = (int)(0xffffffffu - (uint32_t)list[k]);
            }
            __syncthreads();
        } else {
            __syncthreads();
            select_by_histogram<VEC, THREADS>(sm, row, V, K, ntiles);
        }
        for (int k = tid; k < K; k += THREADS) sm.ek[k] = expf(val_of_key(sm.cand_key[k]) - lmax);
        __syncthreads();
        if (wid == 0) {
            float p = 0.f;
            for (int k = lane; k < K; k += 32) p += sm.ek[k];
            p = warp_sum(p);
            if (lane == 0) sm.sum_k = p;
        }
        __syncthreads();
        const float sum_k = sm.sum_k;
        for (int k = tid; k < K; k += THREADS) {
            float w = sm.ek[k] / sum_k;
            int idx = sm.cand_idx[k];
            if (a.pairs) put_pair(a, rowi, k, idx, w);
            if (a.idx) a.idx[rowi * K + k] = idx;
            if (a.w) a.w[rowi * K + k] = w;
        }
        if (a.pairs)
            for (int k = K + tid; k < a.Kp; k += THREADS) put_pair(a, rowi, k, sm.cand_idx[0], 0.f);
        if (tid == 0) {
            float lse = lmax + logf(sum_all);
            if (a.lse) a.lse[rowi] = lse;
            if (a.zk) a.zk[rowi] = sum_k / sum_all;
            if (a.tokens && (a.logp2 || a.step_exp || a.bits_out)) put_surprisal(a, rowi, row, lse);
        }
        __syncthreads();
    }
}

// ---- rows streamed once, a warp (or a few warps) a row --------------------------------------------
// The row is read from HBM once, straight into registers, by one warp when there are rows enough to
// fill the GPU, by up to 32 warps (4 blocks of a cluster) otherwise; the warps of a row meet only at its
// end, so nothing idles at barriers while others stream.  Per 8 logits and lane: one 16-byte load, a
// packed maximum and the sum of exp relative to a running reference.  For the selection a lane only
// leaves the maximum of every group of logits that it reads (a group: 8 logits, or 32 and a multiple
// of it in long rows; at most 64 a lane) in shared memory.  At the row's end the K-th largest of those
// maxima is the bound: at least K logits reach it, exactly K groups (and ties) hold such logits, and
// only those groups, 2 to 10 % of the row, are read again.  The logits at or above the bound, a few
// more than K, are ordered by counting.  A row with more than kListCap of them (ties) is selected by
// counting passes over the row (slow_select).
// Noting every group that reached a running bound instead, with votes or in columns, took 12000 to
// 13000 instructions for a row of 32000 logits, twice what the sum takes; this takes about 3000.
constexpr int kSlots = 64;                          // group maxima of a row, per lane
constexpr int kCodes = 256;                         // groups that are read again
constexpr int kListCap = 256;                       // logits at or above the bound
constexpr int kFinal = 128;                         // K <= kFinal here
constexpr int kBatch = 4;                           // 16-byte loads a lane has in flight per batch (two batches at a time)
constexpr int kStreamWarps = 8;                     // most warps of a block
constexpr int kMaxCluster = 4;

// CHAINED: the kernel may be resident while the logits are being written.
template <bool CHAINED>
__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
    uint4 r;
    if constexpr (CHAINED) asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
    else asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
    return r;
}
__device__ __forceinline__ __half2 as_half2(uint32_t w) { return *reinterpret_cast<const __half2*>(&w); }
__device__ __forceinline__ uint32_t top2_of(const uint4& r) { return hmax2_bits(hmax2_bits(r.x, r.y), hmax2_bits(r.z, r.w)); }
__device__ __forceinline__ uint4 all4(uint32_t w) { return make_uint4(w, w, w, w); }
constexpr uint32_t kNegInf2 = 0xfc00fc00u, kNoValue2 = 0xffffffffu;         // NaN: reaches no bound, loses every maximum
__device__ __forceinline__ uint32_t top_key(uint32_t top2) { return max(key_of(top2 & 0xffffu), key_of(top2 >> 16)); }
__device__ __forceinline__ uint32_t half_at(const uint4& r, int j) {       // j is a compile-time constant after unrolling
    const uint32_t w = j < 2 ? r.x : j < 4 ? r.y : j < 6 ? r.z : r.w;
    return (j & 1) ? w >> 16 : w & 0xffffu;
}
// Order words: larger = earlier in (key descending, index ascending); 32 bits while indices fit 16.
template <class W>
__device__ __forceinline__ W order_word(uint32_t key, int idx) {
    if constexpr (sizeof(W) == 4) return (key << 16) | (0xffffu - (uint32_t)idx);
    else return ((W)key << 32) | (0xffffffffu - (uint32_t)idx);
}
template <class W>
__device__ __forceinline__ uint32_t key_of_word(W w) { return (uint32_t)(w >> (sizeof(W) * 4)); }
template <class W>
__device__ __forceinline__ int idx_of_word(W w) {
    if constexpr (sizeof(W) == 4) return (int)(0xffffu - (w & 0xffffu));
    else return (int)(0xffffffffu - (uint32_t)w);
}

// First place of this lane among the warp's `mine` items; total to all lanes.
__device__ __forceinline__ int warp_excl_scan(int mine, int lane, int& total) {
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += t;
    }
    total = __shfl_sync(kFull, inc, 31);
    return inc - mine;
}

// A row as head logits up to the first 16-byte boundary, nv whole 16-byte groups, and a tail; with FIXED
// the groups are counted from the row's first logit wherever it lies (no head; `phase` logits behind a
// boundary).
struct RowView {
    const __half* row;
    const uint4* body;
    int V, head, nv, phase;
};
template <bool FIXED = false>
__device__ __forceinline__ RowView row_view(const __half* row, int V) {
    RowView r;
    const uint32_t off = (uint32_t)(reinterpret_cast<uintptr_t>(row) & 15u) >> 1;
    r.row = row; r.V = V;
    r.head = FIXED ? 0 : min((int)((8u - off) & 7u), V);
    r.phase = FIXED ? (int)off : 0;
    r.nv = (V - r.head) >> 3;
    r.body = reinterpret_cast<const uint4*>(row + r.head);
    return r;
}
// Group v of a row whose groups do not start on 16-byte boundaries: out of the two aligned vectors that hold
// it (never outside the row), or logit by logit where one of them reaches beyond the row.
__device__ __forceinline__ uint4 group_across(const RowView& r, int v) {
    uint32_t w[8];
    if (v == 0 || 8 * v + 16 > r.V) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            w[j] = (uint32_t)__half_as_ushort(r.row[8 * v + 2 * j]) | ((uint32_t)__half_as_ushort(r.row[8 * v + 2 * j + 1]) << 16);
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
    const uint4* p = reinterpret_cast<const uint4*>(r.row + (8 * v - r.phase));
    const uint4 lo = p[0], hi = p[1];
    w[0] = lo.x; w[1] = lo.y; w[2] = lo.z; w[3] = lo.w; w[4] = hi.x; w[5] = hi.y; w[6] = hi.z; w[7] = hi.w;
    const uint32_t sh = (r.phase & 1) ? 16u : 0u;
    auto at = [&](int i) { return make_uint4(__funnelshift_r(w[i], w[i + 1], sh), __funnelshift_r(w[i + 1], w[i + 2], sh),
                                             __funnelshift_r(w[i + 2], w[i + 3], sh), __funnelshift_r(w[i + 3], w[i + 4], sh)); };
    return r.phase < 4 ? (r.phase < 2 ? at(0) : at(1)) : (r.phase < 6 ? at(2) : at(3));
}
// Four groups that lie `step` apart, all with both their vectors inside the row: the phase, the same in all
// lanes, is looked at once.
__device__ __forceinline__ void groups_across(const RowView& r, int v, int step, uint4 (&q)[4]) {
    const uint4* p = reinterpret_cast<const uint4*>(r.row + (8 * v - r.phase));
    const uint32_t sh = (r.phase & 1) ? 16u : 0u;
    auto fetch = [&](auto word) {
        constexpr int A = decltype(word)::value;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint4 lo = p[u * step], hi = p[u * step + 1];
            const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
            q[u] = make_uint4(__funnelshift_r(w[A], w[A + 1], sh), __funnelshift_r(w[A + 1], w[A + 2], sh),
                              __funnelshift_r(w[A + 2], w[A + 3], sh), __funnelshift_r(w[A + 3], w[A + 4], sh));
        }
    };
    switch (r.phase >> 1) {
        case 0: fetch(std::integral_constant<int, 0>{}); break;
        case 1: fetch(std::integral_constant<int, 1>{}); break;
        case 2: fetch(std::integral_constant<int, 2>{}); break;
        default: fetch(std::integral_constant<int, 3>{});
    }
}
// The ends of the row as groups -1 (lane 0: the head) and nv (lane 1: the tail) of 8, kNoValue where the
// row is not.
__device__ __forceinline__ uint4 row_ends(const RowView& r, int lane) {
    uint32_t w[4] = {kNoValue2, kNoValue2, kNoValue2, kNoValue2};
    if (lane < 2) {
        const int tail0 = r.head + 8 * r.nv, i0 = lane == 0 ? r.head - 8 : tail0;
        const int b = lane == 0 ? 0 : tail0, e = lane == 0 ? r.head : r.V;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int i = i0 + j;
            if (i >= b && i < e) {
                const uint32_t h = (uint32_t)__half_as_ushort(r.row[i]);
                w[j / 2] = (j & 1) ? (w[j / 2] & 0xffffu) | (h << 16) : (w[j / 2] & 0xffff0000u) | h;
            }
        }
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// Logits of a group that reach h2 (one value in both halves): bits p and 16 + p, the halves of word p.
__device__ __forceinline__ uint32_t reach_mask(const uint4& q, uint32_t h2) {
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
    uint32_t m = 0;
#pragma unroll
    for (int p = 0; p < 4; ++p) m |= __hge2_mask(as_half2(w[p]), as_half2(h2)) & (0x10001u << p);
    return m;
}

struct CountShared {                                // of the warps that select a row together
    int count[3], eq[kStreamWarps], n;
};
// Exact selection by counting passes over the row in memory, by the warps of a row's first block (SHARE) or
// one warp: bisection of the K-th largest key between `lo` (at least K logits reach it) and the maximum, then
// the K elements, equal keys in index order, into the list (packed); returns how many there are.  For rows
// whose ties overflow the lists (few finite logits, quantised logits) and rows with few more groups than
// K.  A pass costs ten instructions per 8 logits; NaN reaches nothing.  (40 finite logits of 128256, one row:
// 875 us when one warp passed over it key by key, now 76; 1024 such rows: 1326, 311.)
template <bool SHARE, class W>
__device__ __noinline__ int select_by_count(const __half* row, int V, int K, uint32_t lo, uint32_t kmax, W* list, CountShared& sh, int tw, int tws,
                                            int lane) {
    const RowView r = row_view(row, V);
    const uint4 ends = row_ends(r, lane);
    auto sync = [&]() { if (SHARE) __syncthreads(); else __syncwarp(); };
    if (SHARE) {
        if (tw == 0 && lane < 3) sh.count[lane] = 0;
        if (tw == 0 && lane == 0) sh.n = 0;
        __syncthreads();
    }
    int phase = 0;
    auto count = [&](uint32_t key) {
        const uint32_t h2 = bits_of_key(key) * 0x10001u;
        int c = tw == 0 ? __popc(reach_mask(ends, h2)) : 0;
#pragma unroll 4
        for (int v = tw * 32 + lane; v < r.nv; v += 32 * tws) c += __popc(reach_mask(r.body[v], h2));
        c = __reduce_add_sync(kFull, c);
        if (SHARE) {                                                     // three counters in turn: the one read last is zeroed for the pass after the next
            if (lane == 0) atomicAdd(&sh.count[phase], c);
            __syncthreads();
            c = sh.count[phase];
            phase = phase == 2 ? 0 : phase + 1;
            if (tw == 0 && lane == 0) sh.count[phase == 2 ? 0 : phase + 1] = 0;
        }
        return c;
    };
    uint32_t hi = kmax + 1;                                              // nothing reaches it
    int at_lo = -1, at_hi = 0;                                           // logits that reach lo (-1: not counted), hi
#pragma unroll 1
    for (bool first = true; hi - lo > 1; first = false) {
        const uint32_t mid = first ? lo + 1 : lo + ((hi - lo) >> 1);     // most often the bound itself is the key
        const int c = count(mid);
        if (c >= K) { lo = mid; at_lo = c; } else { hi = mid; at_hi = c; }
    }
    const uint32_t ge2 = bits_of_key(lo) * 0x10001u, gt2 = bits_of_key(lo + 1) * 0x10001u;   // hi = lo + 1 (past +inf: a NaN, which nothing reaches)
    const int need = K - at_hi;                                          // of those equal to lo, in index order
    const bool ranked = at_lo != K;                                      // else all of them
    // a warp takes consecutive groups, the first the head of the row, the last its tail
    const int seg = ((r.nv + tws - 1) / tws + 31) & ~31, v0 = min(tw * seg, r.nv), v1 = min(v0 + seg, r.nv);
    int before = 0, n = 0;                                               // equal ones ahead; elements written (not SHARE)
    if (SHARE && ranked) {
        int e = tw == 0 && lane == 0 ? __popc(reach_mask(ends, ge2) & ~reach_mask(ends, gt2)) : 0;
#pragma unroll 4
        for (int v = v0 + lane; v < v1; v += 32) { const uint4 q = r.body[v]; e += __popc(reach_mask(q, ge2) & ~reach_mask(q, gt2)); }
        e = __reduce_add_sync(kFull, e);
        if (lane == 0) sh.eq[tw] = e;
        __syncthreads();
        for (int w = 0; w < tw; ++w) before += sh.eq[w];
    }
    auto take = [&](const uint4& q, int v) {                             // a group a lane, in index order over the lanes
        const uint32_t ge = reach_mask(q, ge2);
        if (!__any_sync(kFull, ge != 0)) return;
        uint32_t got = reach_mask(q, gt2), eq = ge & ~got;
        if (ranked) {
            int all;
            int rank = before + warp_excl_scan(__popc(eq), lane, all);
            before += all;
#pragma unroll
            for (int j = 0; j < 8; ++j) {                                // word j / 2, half j & 1: index order
                const uint32_t bit = 1u << ((j >> 1) + 16 * (j & 1));
                if (eq & bit) { if (rank < need) got |= bit; ++rank; }
            }
        } else {
            got |= eq;
        }
        int all;
        int at = warp_excl_scan(__popc(got), lane, all);
        int base = n;
        if (SHARE) {
            if (lane == 0) base = atomicAdd(&sh.n, all);
            base = __shfl_sync(kFull, base, 0);
        }
        n += all; at += base;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (got & (1u << ((j >> 1) + 16 * (j & 1)))) {
                if (at < K) list[at] = order_word<W>(key_of(half_at(q, j)), r.head + 8 * v + j);
                ++at;
            }
    };
    if (tw == 0 && r.head > 0) take(lane == 0 ? ends : all4(kNoValue2), -1);
#pragma unroll 1
    for (int v = v0; v < v1; v += 32) take(v + lane < v1 ? r.body[v + lane] : all4(kNoValue2), v + lane);
    if (tw == tws - 1) take(lane == 1 ? ends : all4(kNoValue2), r.nv);
    sync();
    return min(SHARE ? sh.n : n, K);
}

// Orders a list of n words into `sorted`: a word's place is the number of larger ones, which the team's
// lanes count together, 16 bytes of the list at a time.
template <class W, class Sync>
__device__ __forceinline__ void order_list(W* list, int n, W* sorted, int tid, int threads, Sync&& sync) {
    constexpr int PER = 16 / sizeof(W);
    const int pad = (n + PER - 1) & ~(PER - 1);
    if (n + tid < pad) list[n + tid] = 0;                                 // larger than nothing
    sync();
#pragma unroll 1
    for (int i = tid; i < n; i += 3 * threads) {                          // three words a pass: lists are a few words longer than K
        const int i2 = i + threads, i3 = i + 2 * threads;
        const W w1 = list[i], w2 = i2 < n ? list[i2] : (W)0, w3 = i3 < n ? list[i3] : (W)0;
        int rank1 = 0, rank2 = 0, rank3 = 0;
        auto count = [&](W o) { rank1 += o > w1; rank2 += o > w2; rank3 += o > w3; };
#pragma unroll 2
        for (int j = 0; j < pad; j += PER) {
            const uint4 o = *reinterpret_cast<const uint4*>(list + j);
            if constexpr (sizeof(W) == 4) { count(o.x); count(o.y); count(o.z); count(o.w); }
            else { count((W)o.y << 32 | o.x); count((W)o.w << 32 | o.z); }
        }
        sorted[rank1] = w1;
        if (i2 < n) sorted[rank2] = w2;
        if (i3 < n) sorted[rank3] = w3;
    }
    sync();
}
// Writes the row's K selected from the ordered list (one warp).
template <class W>
__device__ __forceinline__ void emit_selected(const TopkArgs& a, long long rowi, const W* sorted, float lmax, float sum_all, int lane) {
    constexpr int R = kFinal / 32;
    const int K = a.K;
    W v[R];
    float ek[R], p = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        v[r] = r * 32 + lane < K ? sorted[r * 32 + lane] : (W)0;
        ek[r] = r * 32 + lane < K ? expf(val_of_key(key_of_word<W>(v[r])) - lmax) : 0.f;
        if (r * 32 + lane < K) p += ek[r];
    }
    const float sum_k = warp_sum(p);
    const int idx0 = __shfl_sync(kFull, idx_of_word<W>(v[0]), 0);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int k = r * 32 + lane;
        if (k < K) {
            const float w = ek[r] / sum_k;
            const int idx = idx_of_word<W>(v[r]);
            if (a.pairs) put_pair(a, rowi, k, idx, w);
            if (a.idx) a.idx[rowi * K + k] = idx;
            if (a.w) a.w[rowi * K + k] = w;
        }
    }
    if (a.pairs)
        for (int k = K + lane; k < a.Kp; k += 32) put_pair(a, rowi, k, idx0, 0.f);
    if (a.zk && lane == 0) a.zk[rowi] = sum_k / sum_all;
}

struct StreamShared {                               // of the warps that share a row (the first block's copy counts)
    float ref[kStreamWarps * kMaxCluster], sum[kStreamWarps * kMaxCluster];
    uint32_t key[kStreamWarps * kMaxCluster];
    int n_codes, n_list;                            // running totals of the end of the row, which the first block's warps share
    uint32_t theta;                                 // its bound
    CountShared by_count;
};
static_assert(kStreamWarps * kMaxCluster <= 32, "a lane for every warp of a row");

// The row after `rowi` (stride: the rows in work at a time) inside its session's position range, or N.
__device__ __forceinline__ long long next_row(const TopkArgs& a, long long rowi, long long stride) {
    for (; rowi < a.N; rowi += stride) {
        if (!(a.pos_begin || a.pos_end)) return rowi;
        const int s = (int)(rowi / a.n_per_session), i = (int)(rowi % a.n_per_session);
        const int b = a.pos_begin ? a.pos_begin[s] : 0, e = a.pos_end ? a.pos_end[s] : a.n_per_session;
        if (i >= b && i < e) return rowi;
    }
    return a.N;
}

// Shared memory of a row: group maxima (binary16, two slots a word), groups to read again, the list.
template <class W>
constexpr size_t stream_smem_per_row() { return 32 * kSlots * 2 + kCodes * 2 + kListCap * sizeof(W); }

__device__ __forceinline__ uint32_t cluster_blocks() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Generic address of the cluster's first block's copy of a shared-memory object.
template <class T>
__device__ __forceinline__ T* at_first_block(T* p) {
    T* r;
    asm("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(p), "r"(0u));
    return r;
}

// Maximum and sum of exp(l - reference) of what a warp reads of a row.
struct RowSum {
    uint32_t m2, lim2;
    float ref, nb;
    unsigned long long s0, s1;
    // A logit more than 4 above the reference moves it, so that no exponent is large (its rounding would
    // show in the sum).
    __device__ __forceinline__ void refer(float to) {
        ref = to; nb = -to * 1.44269504088896341f;
        const uint32_t b = (uint32_t)__half_as_ushort(__float2half_ru(to + 4.0f));
        lim2 = b | (b << 16);
    }
    __device__ __forceinline__ void add_group(const uint4& q) {
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
        const unsigned long long l2e = pack2(1.44269504088896341f, 1.44269504088896341f), nb2 = pack2(nb, nb);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = __half22float2(as_half2(w[j]));
            float x, y, ex, ey;
            unpack2(fma2(pack2(f.x, f.y), l2e, nb2), x, y);
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ex) : "f"(x));
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ey) : "f"(y));
            if (j & 1) s1 = add2(s1, pack2(ex, ey)); else s0 = add2(s0, pack2(ex, ey));
        }
    }
    // The first batch gives the reference; the row's ends are added.
    __device__ __forceinline__ void begin(const uint4 (&first)[kBatch], const uint4& ends, bool has_ends) {
        m2 = kNegInf2;
        if (has_ends) m2 = hmax2_bits(m2, top2_of(ends));
#pragma unroll
        for (int u = 0; u < kBatch; ++u) m2 = hmax2_bits(m2, top2_of(first[u]));
        refer(fmaxf(val_of_key(__reduce_max_sync(kFull, top_key(m2))), -65504.0f));
        s0 = s1 = 0ull;
        if (has_ends) {
            auto real = [](uint32_t w) { const uint32_t m = __vcmpeq2(w, kNoValue2); return (w & ~m) | (kNegInf2 & m); };
            add_group(make_uint4(real(ends.x), real(ends.y), real(ends.z), real(ends.w)));
        }
    }
    // Returns the batch's maximum, top[]: its groups'.
    __device__ __forceinline__ uint32_t add(const uint4 (&q)[kBatch], uint32_t (&top)[kBatch]) {
        uint32_t top4 = kNegInf2;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) { top[u] = top2_of(q[u]); top4 = hmax2_bits(top4, top[u]); }
        m2 = hmax2_bits(m2, top4);
        if (__any_sync(kFull, !__hble2(as_half2(top4), as_half2(lim2)))) {             // a logit above the limit
            const float to = val_of_key(__reduce_max_sync(kFull, top_key(top4)));
            const float f = expf(ref - to);
            const unsigned long long ff = pack2(f, f), z = 0ull;
            s0 = fma2(s0, ff, z); s1 = fma2(s1, ff, z);
            refer(to);
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) add_group(q[u]);
        return top4;
    }
    __device__ __forceinline__ uint32_t max_key() const { return __reduce_max_sync(kFull, top_key(m2)); }
    __device__ __forceinline__ float total() const {
        float x0, x1, x2, x3;
        unpack2(s0, x0, x1); unpack2(s1, x2, x3);
        return warp_sum((x0 + x1) + (x2 + x3));
    }
};

// The selected of a row whose maxima lie in `slots` (NW * ns a lane, `wide` batches each; 0: a group each), by the tws warps
// of a block (SHARE) or by one.  ACROSS: rows may lie off 16-byte boundaries with their groups counted from the
// first logit.
template <bool SHARE, bool ACROSS, class W, class Read>
__device__ __forceinline__ void select_row(const TopkArgs& a, long long rowi, const RowView& r, int NW, int ns, int wide, bool fine, uint32_t* slots, uint16_t* codes, W* list,
                                           W* sorted, StreamShared& local_sh, int tw, int tws, uint32_t kmax, float lmax, float sum_all, int lane, Read&& read) {
    const int K = a.K;
    auto sync = [&]() { if (SHARE) __syncthreads(); else __syncwarp(); };
    // With three quarters as many selected as there are groups the bound holds back little: the logits are
    // counted instead (V = 256, K = 64, 32768 rows: 438 -> 120 us).
    const bool few_groups = fine && 4 * K > 3 * r.nv;
    uint32_t theta = kKeyNegInf;
    int n = 0;
    bool counted = few_groups;
    if (few_groups) read();
    if (!few_groups) {
        // The bound: the K-th largest group maximum (any value that exactly K of them reach will do), searched
        // by one warp with all maxima in its registers.  The search is a chain of ten steps or so: shared among
        // eight warps a step cost 1300 cycles (guards, a shared counter, a barrier), 14400 of the 34000 cycles of a
        // row of 128256 logits by itself; now 5350 of 22000.
        const int S = NW * ns, words = (S + 1) >> 1;
        uint32_t mx[kSlots / 2];                                                      // two maxima each
        if (tw == 0) {
            if (S & 1) reinterpret_cast<uint16_t*>(slots)[(S >> 1) * 64 + lane * 2 + 1] = 0xffffu;   // reaches nothing
            __syncwarp();
#pragma unroll
            for (int i = 0; i < kSlots / 2; ++i) mx[i] = i < words ? slots[i * 32 + lane] : kNoValue2;
            read();
            auto reach = [&](uint32_t h2, auto first) {                               // of this lane's first words
                constexpr int A = SHARE ? 4 : 1;                                      // one sum where other rows fill the gaps
                __half2 c[A];
#pragma unroll
                for (int i = 0; i < A; ++i) c[i] = __float2half2_rn(0.f);
#pragma unroll
                for (int i = 0; i < decltype(first)::value; ++i) c[i % A] = __hadd2(c[i % A], __hge2(as_half2(mx[i]), as_half2(h2)));
                if constexpr (A > 1) c[0] = __hadd2(__hadd2(c[0], c[1]), __hadd2(c[2], c[3]));
                return __half2int_rn(__hadd(__low2half(c[0]), __high2half(c[0])));
            };
            uint32_t hi = kmax + 1, down = 256;                                       // first downwards from the maximum, then between
#pragma unroll 1
            while (hi - theta > 1) {
                const uint32_t mid = down && kmax - theta > down ? kmax - down : theta + ((hi - theta) >> 1), h2 = bits_of_key(mid) * 0x10001u;
                const int c = __reduce_add_sync(kFull, words <= 8 ? reach(h2, std::integral_constant<int, 8>{})
                                                                  : reach(h2, std::integral_constant<int, kSlots / 2>{}));
                if (c >= K) { theta = mid; down = 0; } else { hi = mid; down *= 4; }
                if (c == K) break;
            }
            if (SHARE && lane == 0) local_sh.theta = theta;
        }
        sync();
        if (SHARE) theta = local_sh.theta;
        // Places for a warp's items among the team's: `before` of this lane's first, from a running total.
        auto place = [&](int mine, int* shared_total, int& total) {
            int all;
            int at = warp_excl_scan(mine, lane, all);
            int base = total;
            if (SHARE) {
                if (lane == 0) base = atomicAdd(shared_total, all);
                base = __shfl_sync(kFull, base, 0);
            }
            total += all;                                                             // SHARE: of this warp only
            return base + at;
        };
        // The groups that reach it.
        const uint32_t th2 = bits_of_key(theta) * 0x10001u;
        int n_codes = 0;
        uint32_t hits[2] = {0u, 0u};                                                  // bits i, 16 + i: the maxima of word i (of 16 + i)
        auto hit = [&](uint32_t w, int i) { return __hge2_mask(as_half2(w), as_half2(th2)) & (0x10001u << (i & 15)); };
        if (SHARE) {                                                                  // two warps at least: 16 words at most
#pragma unroll 4
            for (int i = 0; tw + i * tws < words; ++i) hits[0] |= hit(slots[(tw + i * tws) * 32 + lane], i);
        } else {
#pragma unroll
            for (int i = 0; i < kSlots / 2; ++i) hits[i >> 4] |= hit(mx[i], i);
        }
        int at = place(__popc(hits[0]) + __popc(hits[1]), &local_sh.n_codes, n_codes);
#pragma unroll
        for (int h = 0; h < 2; ++h)
            for (uint32_t m = hits[h]; m; m &= m - 1) {
                const int b = __ffs(m) - 1, i = tw + (16 * h + (b & 15)) * tws;
                if (at < kCodes) codes[at] = (uint16_t)((2 * i + (b >> 4)) * 32 + lane);
                ++at;
            }
        sync();
        if (SHARE) n_codes = local_sh.n_codes;
        if (n_codes <= kCodes) {
            // their logits at or above the bound; head and tail of the row are a turn of the last warp's own.  A
            // lane takes one batch of a group where warps share the row (turns are memory latencies: 1700 cycles
            // each), else all of a group (where rows fill the GPU the lanes' divisions cost more than a turn).
            const int steps = fine ? 1 : wide, items = SHARE ? n_codes * steps : n_codes;
            const bool ends_turn = tw == tws - 1 && (r.head > 0 || r.head + 8 * r.nv < r.V);
#pragma unroll 1
            for (int i0 = tw * 32 - (ends_turn ? 32 * tws : 0); i0 < items; i0 += 32 * tws) {
                const bool mine = i0 >= 0 && i0 + lane < items;
                const int ci = !mine ? 0 : SHARE ? (i0 + lane) / steps : i0 + lane, first = SHARE && mine ? i0 + lane - ci * steps : 0;
                const int code = mine ? codes[ci] : 0, sl = code >> 5, w = sl / ns, ls = sl - w * ns;
                const int turns = SHARE || i0 < 0 ? 1 : steps;
#pragma unroll 1
                for (int st = first; st < first + turns; ++st) {
                    const int t = fine ? ls >> 2 : ls * wide + st;
                    const int vb = w * 32 + (code & 31) + (t * kBatch + (fine ? ls & 3 : 0)) * 32 * NW;
                    uint4 q[kBatch];
#pragma unroll
                    for (int u = 0; u < kBatch; ++u) {
                        const int v = vb + u * 32 * NW;
                        q[u] = mine && v < r.nv && !(fine && u) ? (ACROSS && r.phase ? group_across(r, v) : SHARE ? r.body[v] : __ldg(r.body + v)) : all4(kNoValue2);
                    }
                    if (i0 < 0) q[0] = row_ends(r, lane);
                    uint32_t m = 0;                                                    // bits p, 16 + p: the halves of word p
#pragma unroll
                    for (int u = 0; u < kBatch; ++u) {
                        const uint32_t w4[4] = {q[u].x, q[u].y, q[u].z, q[u].w};
#pragma unroll
                        for (int j = 0; j < 4; ++j) m |= __hge2_mask(as_half2(w4[j]), as_half2(th2)) & (0x10001u << (4 * u + j));
                    }
                    for (int to = place(__popc(m), &local_sh.n_list, n); m; m &= m - 1, ++to) {
                        const int b = __ffs(m) - 1, u = (b >> 2) & 3;
                        const int v = i0 >= 0 ? vb + u * 32 * NW : lane == 0 ? -1 : r.nv;
                        const int e = r.head + 8 * v + 2 * (b & 3) + (b >> 4);
                        if (to < kListCap) list[to] = order_word<W>(key_of(__half_as_ushort(SHARE ? r.row[e] : __ldg(r.row + e))), e);   // a first-level hit
                    }
                }
            }
        }
        sync();
        if (SHARE) n = local_sh.n_list;
        counted = n_codes > kCodes || n > kListCap;
    }
    if (counted) {
        sync();                                                                   // all have read the totals
        n = select_by_count<SHARE, W>(r.row, r.V, K, theta, kmax, list, local_sh.by_count, tw, tws, lane);
    }
    order_list<W>(list, n, sorted, SHARE ? (int)threadIdx.x : lane, tws * 32, sync);
    if (tw == 0) {
        // NaN logits reach no bound: a row with fewer than K others is filled up with candidate 0 at weight 0
        for (int i = n + lane; i < K; i += 32) sorted[i] = order_word<W>(kKeyNegInf, 0);
        __syncwarp();
        emit_selected<W>(a, rowi, sorted, lmax, sum_all, lane);
    }
}

// SHARE: the warps of a cluster of blocks (of a block, if it is alone) share a row; otherwise every warp
// has a row of its own.
// FIXED: the order in which a row's exponentials are added depends on V alone, not on how many rows the call
// has or where the row lies in memory.  The adaptive step (Def. 7) floors a multiple of the row's
// log-sum-exp, so a batch encoded at once and restored a session at a time must find the same bits.  The
// row is cut into parts of its own (row_parts), a warp takes one after another, and groups are counted
// from the row's first logit.
// (1: all rows start on a 16-byte boundary; 2: any rows; the same sums.)
template <bool SELECT, bool SHARE, int FIXED, class W>
__global__ void __launch_bounds__(32 * kStreamWarps, 4) topk_stream_kernel(const TopkArgs a) {
    extern __shared__ __align__(16) unsigned char stream_raw[];
    __shared__ StreamShared local_sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int blocks = SHARE ? (int)cluster_blocks() : 1;
    const int warps = SHARE ? nwarps * blocks : 1, wfirst = SHARE ? (int)cluster_rank() * nwarps + warp : 0;   // warps of the row, this one's number
    const int NW = FIXED ? a.parts : warps;                                              // parts of the row: one a warp, or several
    StreamShared& sh = *(SHARE && blocks > 1 ? at_first_block(&local_sh) : &local_sh);
    auto meet = [&]() {
        if (blocks > 1) {
            asm volatile("barrier.cluster.arrive.release;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        } else {
            __syncthreads();
        }
    };
    unsigned char* raw = stream_raw + (SHARE ? 0 : (size_t)warp * stream_smem_per_row<W>());
    uint32_t* slots = reinterpret_cast<uint32_t*>(raw);                                  // [kSlots / 2][32]
    uint16_t* codes = reinterpret_cast<uint16_t*>(slots + 16 * kSlots);
    W* list = reinterpret_cast<W*>(codes + kCodes);
    uint16_t* my_slots = reinterpret_cast<uint16_t*>(SHARE && blocks > 1 ? at_first_block(slots) : slots);
    if (SHARE && blocks > 1) meet();                                                      // all blocks of the cluster have started
    chain_next();
    chain_wait();
    zero_tickets(a);
    const long long group = SHARE ? blockIdx.x / blocks : (long long)blockIdx.x * nwarps + warp;
    const long long stride = SHARE ? gridDim.x / blocks : (long long)gridDim.x * nwarps;

    for (long long rowi = next_row(a, group, stride); rowi < a.N; rowi = next_row(a, rowi + stride, stride)) {
        const RowView r = row_view<FIXED != 0>(a.logits + rowi * (long long)a.V, a.V);
        auto fetch = [&](int v) { return FIXED == 2 && r.phase ? group_across(r, v) : ld_stream<SHARE>(r.body + v); };
        const int per = kBatch * 32 * NW, batches = max(1, (r.nv + per - 1) / per);
        // Slots of this warp: one a group of 8 where all the row's fit, else one for every `wide` batches.
        const bool fine = NW * batches * kBatch <= kSlots;
        const int wide = (NW * batches + kSlots - 1) / kSlots, ns = fine ? batches * kBatch : (batches + wide - 1) / wide;
        uint32_t part_key = 0;                                                            // FIXED: lane p holds part p
        float part_ref = 0.f, part_sum = 0.f;
        uint32_t kmax = 0;
        float ref = 0.f, sum_all = 0.f;
        auto load = [&](int w, int t, uint4 (&q)[kBatch]) {                               // group u of batch t of part w
            const int at = w * 32 + lane + t * per;
            if (FIXED == 2 && r.phase && w + t > 0 && (t + 1) * per < r.nv) {
                groups_across(r, at, 32 * NW, q);
            } else if ((FIXED != 2 || !r.phase) && (t + 1) * per <= r.nv) {
#pragma unroll
                for (int u = 0; u < kBatch; ++u) q[u] = ld_stream<SHARE>(r.body + at + u * 32 * NW);
            } else {
#pragma unroll
                for (int u = 0; u < kBatch; ++u) q[u] = at + u * 32 * NW < r.nv ? fetch(at + u * 32 * NW) : all4(kNegInf2);
            }
        };
        int wrow = wfirst, wload = wfirst, tload = 0;
        auto load_next = [&](uint4 (&q)[kBatch]) {                                        // FIXED: on into the next part of this warp
            load(wload, tload, q);
            if (++tload == batches && wload + warps < NW) { tload = 0; wload += warps; }
        };
        uint4 cur[kBatch], nxt[kBatch];
        if (FIXED) { load_next(cur); load_next(nxt); }
        else { load(wrow, 0, cur); load(wrow, 1, nxt); }
#pragma unroll 1
        do {
            const bool has_ends = wrow == 0 && (r.head > 0 || r.head + 8 * r.nv < r.V);
            const uint4 ends = has_ends ? row_ends(r, lane) : all4(kNoValue2);
            RowSum sum;
            sum.begin(cur, ends, has_ends);
            // slot s of a lane: half s & 1 of word (s / 2, lane)
            auto put_slot = [&](int slot, uint32_t top2) {
                const int sl = wrow * ns + slot;
                my_slots[(sl >> 1) * 64 + lane * 2 + (sl & 1)] = (uint16_t)hmax2_bits(top2, top2 >> 16);   // the low half: of both
            };
            uint32_t top[kBatch];
            uint32_t group2 = kNegInf2;                                                       // of the slot being filled
            int left = wide, slot = 0;
            auto filled = [&](uint32_t top4) {
                group2 = hmax2_bits(group2, top4);
                if (--left == 0) { put_slot(slot++, group2); group2 = kNegInf2; left = wide; }
            };
            if (FIXED == 2 || (SELECT && fine)) {
#pragma unroll 1
                for (int t = 0; t < batches; ++t) {
                    const uint32_t top4 = sum.add(cur, top);
                    if (FIXED == 2 && !fine) filled(top4);
#pragma unroll
                    for (int u = 0; u < kBatch; ++u) {
                        if (FIXED != 2 || fine) put_slot(t * kBatch + u, top[u]);
                        cur[u] = nxt[u];
                    }
                    if (FIXED) load_next(nxt);
                    else load(wrow, t + 2, nxt);
                }
                if (FIXED == 2 && !fine && left != wide) put_slot(slot, group2);
            } else {
#pragma unroll 1
                for (int t = 0; t < batches; t += 2) {
                    const uint32_t t0 = sum.add(cur, top);
                    if (SELECT) filled(t0);
                    if (FIXED) load_next(cur);
                    else load(wrow, t + 2, cur);
                    if (t + 1 < batches) {
                        const uint32_t t1 = sum.add(nxt, top);
                        if (SELECT) filled(t1);
                        if (FIXED) load_next(nxt);
                    } else if (FIXED) {                                                       // the next part begins with what lies in nxt
#pragma unroll
                        for (int u = 0; u < kBatch; ++u) { const uint4 q = cur[u]; cur[u] = nxt[u]; nxt[u] = q; }
                    }
                    if (!FIXED) load(wrow, t + 3, nxt);
                }
                if (SELECT && left != wide) put_slot(slot, group2);
            }

            // Maximum and sum of the part, then of the row.
            kmax = sum.max_key();
            ref = sum.ref;
            sum_all = sum.total();
            if (SHARE) {
                if (lane == 0) { sh.key[wrow] = kmax; sh.ref[wrow] = ref; sh.sum[wrow] = sum_all; }
            } else if (FIXED && lane == wrow) {
                part_key = kmax; part_ref = ref; part_sum = sum_all;
            }
        } while (FIXED && (wrow += warps) < NW);
        float lmax;
        if (SHARE || FIXED) {
            const bool on = lane < NW;                                                    // a lane a part of the row
            if (SHARE) {
                if (SELECT && wfirst == 0 && lane == 0) sh.n_codes = sh.n_list = 0;
                meet();
                if (on) { part_key = sh.key[lane]; part_ref = sh.ref[lane]; part_sum = sh.sum[lane]; }
            }
            kmax = __reduce_max_sync(kFull, on ? part_key : 0u);
            lmax = val_of_key(kmax);
            sum_all = warp_sum(on ? part_sum * expf(part_ref - lmax) : 0.f);
        } else {
            lmax = val_of_key(kmax);
            sum_all *= expf(ref - lmax);
        }

        if (SELECT && (!SHARE || wfirst < nwarps))                                        // the row's own warp, or all warps of the first block
            select_row<SHARE, FIXED == 2, W>(a, rowi, r, NW, ns, wide, fine, slots, codes, list,
                                             reinterpret_cast<W*>(slots), local_sh, SHARE ? warp : 0, SHARE ? nwarps : 1, kmax, lmax, sum_all, lane, []() {});
        if (lane == 0 && wfirst == 0) put_row(a, rowi, r.row, lmax + logf(sum_all));
        __syncwarp();
        if (SHARE) meet();                                                                // the row's shared state is free again
    }
}

// Long rows, many of them: a block an SM, in which teams of warps stream rows (a row's parts to a team's warps) and
// other warps select from the rows that have passed, so that the end of a row (the bound's search, a second
// look at a few groups, the ordering: 12000 cycles for a warp, chains for the most part) takes place under the
// streaming of the next rows.  With a warp a row all of them reach their ends together, and memory idles meanwhile.
// The block's rows (blockIdx, + gridDim, ...; those inside the position ranges) are numbered q = 0, 1, ...: team
// q % teams streams row q into buffer q % kFinishers, which the finishing warp of that number reads.  Full and
// empty buffers are hardware barriers (the waiting side sleeps); the number of teams divides the number of
// buffers, so that a buffer belongs to one team and its barrier's generations cannot mix.  A buffer of a team of 4
// is free again as soon as the finishing warp has its maxima in registers; teams of 8 have time, and 16 KB more L1 are
// worth more (4096 rows of 128256: 204 us, 191).
// The logits come through a ring in shared memory that every lane fills for itself, asynchronously (held in
// registers across rows they were spilled: 4096 rows of 128256 434 us).
// What bounds it: the streaming warps' latency a batch (1700 to 2000 cycles, 16 warps, 130 KB in flight an SM).
// 4000 rows of 128256, K = 64, every output: 270 -> 191 us (idx and w only 263, 186; without a selection 168, the copy
// rate 156); 16384 rows of 32000: 268 -> 242.
constexpr int kStreamers = 16, kFinishers = 8, kMostTeam = 8;           // warps of a block: streaming, finishing; most of a team
constexpr int kRing = 4;                                                // batches of a warp on their way
static_assert(2 * kFinishers <= 16, "a block has 16 barriers");
template <int TEAM, class W>
struct __align__(16) PipeRow {
    static constexpr bool kEarly = TEAM < 8;                            // see above
    uint32_t slots[16 * kSlots];
    uint16_t codes[kCodes];
    W list[kEarly ? 2 * kListCap : kListCap];
    float ref[kMostTeam], sum[kMostTeam];
    uint32_t key[kMostTeam];
    __device__ __forceinline__ W* sorted() { return kEarly ? list + kListCap : reinterpret_cast<W*>(slots); }
};
template <int TEAM>
__device__ __forceinline__ void wait_barrier(int id) { asm volatile("barrier.sync %0, %1;" ::"r"(id), "n"(32 * (TEAM + 1)) : "memory"); }
template <int TEAM>
__device__ __forceinline__ void arrive_barrier(int id) { asm volatile("barrier.arrive %0, %1;" ::"r"(id), "n"(32 * (TEAM + 1)) : "memory"); }

// The block's rows of numbers first, first + step, ...
struct PipeRows {
    long long at;
    int q, step;
    __device__ __forceinline__ PipeRows(const TopkArgs& a, int first, int step_) : at(next_row(a, blockIdx.x, gridDim.x)), q(0), step(step_) { skip(a, first); }
    __device__ __forceinline__ void skip(const TopkArgs& a, int rows) {
        if (a.pos_begin || a.pos_end) {
            for (int i = 0; i < rows && at < a.N; ++i) at = next_row(a, at + gridDim.x, gridDim.x);
        } else {
            at += (long long)rows * gridDim.x;
        }
        q += rows;
    }
    __device__ __forceinline__ void next(const TopkArgs& a) { skip(a, step); }
};
constexpr int kPipeLeast = 24576;                                       // shortest row
template <int TEAM>
struct PipeCut {                                                        // a warp's share of a row: a slot every `wide` batches
    int batches, wide, ns;
    __device__ __forceinline__ explicit PipeCut(int nv) {
        constexpr int per = kBatch * 32 * TEAM;
        static_assert((kPipeLeast - 7) / 8 * kBatch * TEAM > kSlots * per, "more groups than slots");
        batches = (nv + per - 1) / per;
        wide = (TEAM * batches + kSlots - 1) / kSlots;
        ns = (batches + wide - 1) / wide;
    }
};

template <int TEAM, class W>
__device__ __forceinline__ void pipe_stream(const TopkArgs& a, PipeRow<TEAM, W>* rows, uint4* ring, int team, int w, int lane) {
    constexpr int per = kBatch * 32 * TEAM, kTeams = kStreamers / TEAM;
    static_assert(kFinishers % kTeams == 0, "a buffer belongs to one team, which meets at its barriers in the order of its rows");
    const int first = w * 32 + lane;                                                          // this lane's first group of a row
    PipeRows to_load(a, team, kTeams), row = to_load;
    // A lane copies what it will read itself: kRing batches of kBatch groups.
    const uint4* src = nullptr;
    int left_nv = 0, into = 0;                                                                // of the row being copied: groups from this lane's next one on
    auto open_row = [&]() {
        if (to_load.at >= a.N) return;
        const RowView r = row_view(a.logits + to_load.at * (long long)a.V, a.V);
        src = r.body + first; left_nv = r.nv - w * 32;
    };
    auto copy_next = [&]() {                                                                  // on into the team's next row
        if (to_load.at < a.N) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(ring + into * (kBatch * 32));
#pragma unroll
            for (int u = 0; u < kBatch; ++u)
                if (lane + u * 32 * TEAM < left_nv)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + u * 512), "l"(src + u * 32 * TEAM) : "memory");
            into = into + 1 == kRing ? 0 : into + 1;
            src += per; left_nv -= per;
            if (left_nv + w * 32 <= 0) { to_load.next(a); open_row(); }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    open_row();
#pragma unroll 1
    for (int i = 0; i < kRing - 1; ++i) copy_next();
    int at = 0;                                                                               // the ring's batch to be read
#pragma unroll 1
    for (; row.at < a.N; row.next(a)) {
        const RowView r = row_view(a.logits + row.at * (long long)a.V, a.V);
        const PipeCut<TEAM> cut(r.nv);
        const int b = row.q % kFinishers;
        PipeRow<TEAM, W>& to = rows[b];
        auto put_slot = [&](int slot, uint32_t top2) {                                        // slot s of a lane: half s & 1 of word (s / 2, lane)
            const int sl = w * cut.ns + slot;
            reinterpret_cast<uint16_t*>(to.slots)[(sl >> 1) * 64 + lane * 2 + (sl & 1)] = (uint16_t)hmax2_bits(top2, top2 >> 16);
        };
        uint32_t group2 = kNegInf2;
        int left = cut.wide, slot = 0;
        const bool has_ends = w == 0 && (r.head > 0 || r.head + 8 * r.nv < r.V);
        const uint4 ends = has_ends ? row_ends(r, lane) : all4(kNoValue2);                    // read now, taken at the row's end
        RowSum sum;
#pragma unroll 1
        for (int t = 0; t < cut.batches; ++t) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");
            uint4 g[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) g[u] = ring[at * (kBatch * 32) + u * 32];
            if ((t + 1) * per > r.nv) {
#pragma unroll
                for (int u = 0; u < kBatch; ++u) if (first + t * per + u * 32 * TEAM >= r.nv) g[u] = all4(kNegInf2);
            }
            at = at + 1 == kRing ? 0 : at + 1;
            copy_next();                                                                      // over the batch before this one
            if (t == 0) {
                sum.begin(g, g[0], false);
                if (row.q >= kFinishers) wait_barrier<TEAM>(kFinishers + b);                        // the row that was there has been read
            }
            uint32_t top[kBatch];
            group2 = hmax2_bits(group2, sum.add(g, top));
            if (--left == 0) { put_slot(slot++, group2); group2 = kNegInf2; left = cut.wide; }
        }
        if (left != cut.wide) put_slot(slot, group2);
        if (has_ends) {
            auto real = [](uint32_t v) { const uint32_t m = __vcmpeq2(v, kNoValue2); return (v & ~m) | (kNegInf2 & m); };
            const uint4 g[kBatch] = {make_uint4(real(ends.x), real(ends.y), real(ends.z), real(ends.w)), all4(kNegInf2), all4(kNegInf2), all4(kNegInf2)};
            uint32_t top[kBatch];
            sum.add(g, top);
        }
        const uint32_t kmax = sum.max_key();
        const float total = sum.total();
        if (lane == 0) { to.key[w] = kmax; to.ref[w] = sum.ref; to.sum[w] = total; }
        __syncwarp();
        arrive_barrier<TEAM>(b);
    }
}
template <int TEAM, class W>
__device__ __forceinline__ void pipe_finish(const TopkArgs& a, PipeRow<TEAM, W>& from, StreamShared& unused, int b, int lane) {
    constexpr bool kEarly = PipeRow<TEAM, W>::kEarly;
    PipeRows row(a, b, kFinishers);
#pragma unroll 1
    while (row.at < a.N) {
        const long long rowi = row.at;
        const RowView r = row_view(a.logits + rowi * (long long)a.V, a.V);
        const PipeCut<TEAM> cut(r.nv);
        row.next(a);
        wait_barrier<TEAM>(b);
        const bool on = lane < TEAM;
        const uint32_t kmax = __reduce_max_sync(kFull, on ? from.key[lane] : 0u);
        const float lmax = val_of_key(kmax);
        const float sum_all = warp_sum(on ? from.sum[lane] * expf(from.ref[lane] - lmax) : 0.f);
        select_row<false, false, W>(a, rowi, r, TEAM, cut.ns, cut.wide, false, from.slots, from.codes, from.list, from.sorted(), unused, 0, 1, kmax, lmax,
                                    sum_all, lane, [&]() { if (kEarly && row.at < a.N) arrive_barrier<TEAM>(kFinishers + b); });   // the next row may be put there
        if (lane == 0) put_row(a, rowi, r.row, lmax + logf(sum_all));
        __syncwarp();
        if (!kEarly && row.at < a.N) arrive_barrier<TEAM>(kFinishers + b);
    }
}
template <int TEAM, class W>
__global__ void __launch_bounds__(32 * (kStreamers + kFinishers), 1) topk_pipe_kernel(const TopkArgs a) {
    extern __shared__ __align__(16) unsigned char pipe_raw[];
    __shared__ StreamShared unused;
    PipeRow<TEAM, W>* rows = reinterpret_cast<PipeRow<TEAM, W>*>(pipe_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, f = warp - kStreamers;
    zero_tickets(a);
    if (f < 0) pipe_stream<TEAM, W>(a, rows, reinterpret_cast<uint4*>(rows + kFinishers) + warp * (kRing * kBatch * 32) + lane, warp / TEAM, warp % TEAM, lane);
    else pipe_finish<TEAM, W>(a, rows[f], unused, f, lane);
}

}  // namespace

// Parts of a row whose sum must not depend on the call (FIXED): a power of two with at least 1024 logits
// each, at most a warp of one block.
static int row_parts(int V) {
    int n = 1;
    while (n < kStreamWarps && 2ll * n * 1024 <= V) n *= 2;
    return n;
}

template <bool SELECT, int FIXED, class W>
static cudaError_t launch_stream(TopkArgs a, int sms, cudaStream_t st, int* few_blocks) {
    // Warps a row, in powers of two, each with at least 1024 logits of its own; one when rows alone fill the
    // GPU.  Up to a block of eight: as many as the GPU holds for all rows (32 a SM).  Up to four blocks (a
    // cluster): only while that is a quarter of the GPU, since a cluster's blocks are placed together
    // (64 rows of 128256, 64 warps each: 51 us; 16 warps: 25; one row: 8 warps 24.6, 32 warps 20.5).
    a.parts = row_parts(a.V);
    const int most = FIXED ? a.parts : kStreamWarps * kMaxCluster;
    int warps = 1;
    while (warps < most && 2ll * warps * 1024 <= a.V &&
           2ll * warps * a.N <= (warps < kStreamWarps ? 32ll : 8ll) * sms) warps *= 2;
    const bool share = warps > 1;
    const int per_block = share ? std::min(warps, kStreamWarps) : kStreamWarps, cluster = share ? warps / per_block : 1;
    const size_t smem = !SELECT ? 0 : stream_smem_per_row<W>() * (share ? 1 : per_block);
    auto kern = share ? topk_stream_kernel<SELECT, true, FIXED, W> : topk_stream_kernel<SELECT, false, FIXED, W>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int occ = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, per_block * 32, smem) != cudaSuccess || occ < 1) occ = 1;
    const long long want = share ? a.N * cluster : (a.N + per_block - 1) / per_block;
    const unsigned blocks = (unsigned)std::min<long long>(want, (long long)sms * occ / cluster * cluster);
    *few_blocks = share || (int)blocks <= sms ? (int)blocks : 0;
    count_launch();
    return launch_kernel(kern, blocks, per_block * 32, smem, st, a.chained && *few_blocks > 0, cluster, a);
}

template <int TEAM, class W>
static cudaError_t launch_pipe(const TopkArgs& a, int sms, cudaStream_t st) {
    const size_t smem = kFinishers * sizeof(PipeRow<TEAM, W>) + (size_t)kStreamers * kRing * kBatch * 32 * sizeof(uint4);
    const cudaError_t e = cudaFuncSetAttribute(topk_pipe_kernel<TEAM, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    count_launch();
    return launch_kernel(topk_pipe_kernel<TEAM, W>, (unsigned)std::min<long long>(a.N, sms), 32 * (kStreamers + kFinishers), smem, st, false, 1, a);
}

// Where topk_pipe_kernel is the quicker one (times of topk_stream_kernel / of teams, idx and w only unless said).
// Long rows, from two an SM on: 300 rows of 32000: 17.6 / 14.6 us, of 128256: 37.7 / 33.0.  A row's costs beside its
// batches weigh more the shorter it is: teams of 4 warps for rows up to 65536 (16384 rows of 32000: 245 us with 8, 223),
// of 8 beyond (4096 rows of 128256: 201 us with 4, 191), and a warp a row for short ones (16384 rows of 16384: 151 us
// against 162).
// More than 64 rows an SM of up to 65536: a warp a row has no last wave to speak of, and teams pay only where the
// ends of rows are long (large K) but not so long against a row that they keep the finishing warps busier than the
// streaming ones.  10000 rows: of 24576 K = 16 102 / 107, 64 135 / 130, 80 140 / 144, 128 167 / 183; of 32000 16 136 / 134, 40 156 /
// 148, 64 168 / 152, 128 206 / 212; of 50001 16 207 / 224, 40 222 / 234, 64 239 / 240, 100 280 / 256; 32768 rows of 32000: 16
// 424 / 457, 64 523 / 505; 8000 rows: of 24576 16 91 / 87, 128 153 / 148.
// With position ranges the rows are counted off one by one, and half of them may be missing: rows beyond 65536 only,
// and from where the other kernel gives a warp a row (both calls with 2 streams of 32, half in range: 4000 rows of
// 32000 152 / 164 us; 3000 rows of 65544 289 / 187, of 128256 406 / 240; 2100 rows of 65544 184 / 180, of 100001 250 /
// 258; 1000 rows of 100001 137 / 144).
static bool teams_pay(const TopkArgs& a, int sms) {
    if (a.V < kPipeLeast || a.N < 2ll * sms) return false;
    if (a.pos_begin || a.pos_end) return a.V > 65536 && a.N > 16ll * sms;
    return a.V > 65536 || a.N <= 64ll * sms || (a.K >= 48 && (a.K < 80 || a.V >= 32000));
}

cudaError_t launch_topk(const TopkArgs& a, cudaStream_t st, int* few_blocks) {
    *few_blocks = 0;
    if (a.N <= 0) return cudaSuccess;
    const int sms = sm_count();
    const bool select = a.pairs || a.idx || a.w || a.zk;
    if (!select) return launch_stream<false, 0, uint32_t>(a, sms, st, few_blocks);
    const bool vec = (a.V % 8 == 0) && ((reinterpret_cast<uintptr_t>(a.logits) & 15) == 0);
    if (a.K <= kFinal) {
        const int fixed = !(a.step_exp || a.bits_out) ? 0 : vec ? 1 : 2;
        // Calls with an adaptive step need sums of the same parts at any number of rows.
        if (!fixed && teams_pay(a, sms)) return a.V <= 65536 ? launch_pipe<4, uint32_t>(a, sms, st) : launch_pipe<8, unsigned long long>(a, sms, st);
        if (a.V <= 65536) return fixed == 0 ? launch_stream<true, 0, uint32_t>(a, sms, st, few_blocks)
                               : fixed == 1 ? launch_stream<true, 1, uint32_t>(a, sms, st, few_blocks) : launch_stream<true, 2, uint32_t>(a, sms, st, few_blocks);
        return fixed == 0 ? launch_stream<true, 0, unsigned long long>(a, sms, st, few_blocks)
             : fixed == 1 ? launch_stream<true, 1, unsigned long long>(a, sms, st, few_blocks) : launch_stream<true, 2, unsigned long long>(a, sms, st, few_blocks);
    }
    // The second pass over a row should find it in L2: rows of up to 128 KB are read by 256 threads
    // with five blocks per SM, longer rows by 512 threads with two blocks per SM (two, so that one
    // block streams while the other sits at the barrier between its passes).
    const bool wide = (long long)a.V * 2 > 128 * 1024;
    auto launch = [&](auto kern, int threads, int cap) {
        int occ = 1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, 0) != cudaSuccess || occ < 1) occ = 1;
        const long long per_sm = occ < cap ? occ : cap;       // the rows in flight stay within L2
        const long long blocks = a.N < sms * per_sm ? a.N : sms * per_sm;
        const bool few = a.N <= sms;
        *few_blocks = few ? (int)blocks : 0;
        count_launch();
        return launch_kernel(kern, (unsigned)blocks, threads, 0, st, a.chained && few, 1, a);
    };
    if (wide) return vec ? launch(topk_softmax_kernel<true, 512>, 512, 2) : launch(topk_softmax_kernel<false, 512>, 512, 2);
    return vec ? launch(topk_softmax_kernel<true, 256>, 256, 5) : launch(topk_softmax_kernel<false, 256>, 256, 5);
}

}  // namespace plc
