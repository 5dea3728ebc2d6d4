// Fused predict / quantise / rANS kernels.
//
// One warp owns one (stream, chunk): it walks the chunk's positions (backwards when encoding,
// forwards when decoding), and for each position
//   1. gathers the K candidate rows of its table with 128-bit loads and accumulates the mixture
//      mu = sum_k w_k T[idx_k] in binary32 (each lane: 8 components of every ROWS-th row, then a
//      shuffle reduce-scatter so that lane l ends with its G = d/32 components),
//   2. derives the scale class from the mixture variance (precomputed row norms),
//   3. quantises the residual (encoder) or adds the decoded residual back (decoder),
//   4. runs one interleaved rANS step per owned component, the 32 lanes sharing one word stream.
// The encoder writes its words back to front into a per-warp staging area (global memory, reused
// from chunk to chunk so it stays in L2), then reserves the chunk's final place with one atomicAdd
// and copies it there.  Work items are handed out by an atomic ticket in table-major order so that
// the warps running at any time gather from few tables.
#include <algorithm>
#include <type_traits>

#include "plc_codec.cuh"

namespace plc {
namespace {

constexpr int kWarpsPerBlock = 8;
constexpr int kThreads = kWarpsPerBlock * 32;
// Blocks per SM.  The coder alone (symbols or predictions read from memory) wants warps: 5, 48 registers.
// The gather wants row loads in flight more than warps: 32 warps at 64 registers hold a stretch of 32
// rows' loads where 40 held 8 (256 streams x 16384 positions, skewed candidates: 6.18 + 6.46 -> 5.49 +
// 5.79 ms), and where the rows come from L2 (one queue for the whole GPU) 24 at 80 are better still:
// fewer tables in flight, more L1 (131072 positions x 32 streams, uniform candidates: decode 7.7 ->
// 6.8 ms).  The gather kernels with a coder are one block an SM, so that its warps share one copy of the
// coder's tables (20 KB) and the L1 is 60 KB larger than with blocks of eight (1024 streams x 16384
// positions, skewed: 21.28 + 20.94 -> 20.51 + 20.21 ms; 131072 positions x 64 streams: decode 14.1 -> 13.6 ms).
constexpr int kBlocksPerSM = 5, kGatherBlocks = 4;
constexpr int kGatherWarps = kGatherBlocks * kWarpsPerBlock, kFarWarps = 24;

// Squared row norms; a warp takes kNormRows rows, whose norms are one sector.
constexpr int kNormRows = 8;
template <int D>
__global__ void __launch_bounds__(256) rownorm_kernel(const __half* __restrict__ T, float* __restrict__ out, long long rows, unsigned int* not_finite) {
    constexpr int G = Geo<D>::G;
    const int lane = threadIdx.x & 31;
    const long long warp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    const int c0 = first_comp<D>(lane);
    for (long long r0 = warp * kNormRows; r0 < rows; r0 += nw * kNormRows) {
        float mine = 0.f;
#pragma unroll 4
        for (int j = 0; j < kNormRows; ++j) {
            if (r0 + j >= rows) break;
            const __half* row = T + (r0 + j) * D + c0;
            float x[G];
#pragma unroll
            for (int g = 0; g < G; ++g) x[g] = __half2float(row[g]);
            const float s = warp_norm2<G>(x);
            if (lane == j) mine = s;
        }
        if (!(mine < __int_as_float(0x7f800000))) *not_finite = 1u;           // squares of finite binary16 values sum to less
        if (lane < kNormRows && r0 + lane < rows) out[r0 + lane] = mine;
    }
}

// by_row[v][t] = norms[t][v], by tiles of 32 x 32.
__global__ void __launch_bounds__(256) norms_by_row_kernel(const float* __restrict__ norms, float* __restrict__ by_row, int V, int tables) {
    __shared__ float tile[32][33];
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5, v0 = blockIdx.x * 32, t0 = blockIdx.y * 32;
    for (int j = y; j < 32; j += 8)
        if (t0 + j < tables && v0 + x < V) tile[j][x] = norms[(long long)(t0 + j) * V + v0 + x];
    __syncthreads();
    for (int j = y; j < 32; j += 8)
        if (v0 + j < V && t0 + x < tables) by_row[(long long)(v0 + j) * tables + t0 + x] = tile[x][j];
}

// Variance terms s1[row][t] = sum_k w_k ||T[t][idx_k]||^2 of every (position, table), ahead of the gather kernels: the
// norms of a candidate lie beside each other for all tables, so a warp reads them for 32 * VEC tables at
// once, where the gather, one table a warp, takes a sector a candidate (64 of its 242 L1 wavefronts a vector).  0.36 ms
// for 1024 tables x 16384 positions, where the gather becomes 1.0 ms shorter.
// The additions are those of predict's own sum and warp_sum (lane l: candidates l, l + 32, ...; then lanes
// l and l ^ 16, l ^ 8, ...), so both give the same bits.  Lanes: `width` of them (a power of two) side by side in
// the tables, 32 / width positions a warp.
template <int VEC>
__global__ void __launch_bounds__(256) variance_kernel(const CodecArgs a, int width, int row_shift, int load_shift) {
    using Vec = std::conditional_t<VEC == 4, float4, float2>;
    const int lane = threadIdx.x & 31, W = 2 * a.sh.L * a.sh.H, Kp = a.sh.Kp, iters = Kp >> load_shift, per_warp = 32 / width;
    const int t0 = ((int)blockIdx.y * width + (lane & (width - 1))) * VEC;
    const long long N = (long long)a.S * a.n, row = ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * per_warp + lane / width;
    if (row >= N || t0 >= W) return;
    if (a.pos_begin || a.pos_end) {
        const int s = (int)(row / a.n), i = (int)(row % a.n);
        if (i < (a.pos_begin ? a.pos_begin[s] : 0) || i >= (a.pos_end ? a.pos_end[s] : a.n)) return;   // no pairs there
    }
    const int2* pairs = a.pairs + row * Kp;
    float stack[5][VEC], sum[VEC];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const int l = (i & 1) * 16 + (i >> 1 & 1) * 8 + (i >> 2 & 1) * 4 + (i >> 3 & 1) * 2 + (i >> 4);
#pragma unroll
        for (int j = 0; j < VEC; ++j) sum[j] = 0.f;
#pragma unroll 2
        for (int k = l; k < Kp; k += 32) {
            const int2 pr = __ldg(pairs + (k & ((1 << load_shift) - 1)) * iters + (k >> load_shift));
            const uint32_t at = (uint32_t)pr.x >> row_shift;
            const Vec n = __ldg(reinterpret_cast<const Vec*>(a.norms_by_row + (size_t)at * W + t0));
            const float w = __int_as_float(pr.y);
            sum[0] = __fmaf_rn(w, n.x, sum[0]); sum[1] = __fmaf_rn(w, n.y, sum[1]);
            if constexpr (VEC == 4) { sum[2] = __fmaf_rn(w, n.z, sum[2]); sum[3] = __fmaf_rn(w, n.w, sum[3]); }
        }
        int level = 0;
#pragma unroll
        for (; level < 5 && (i >> level & 1); ++level)
#pragma unroll
            for (int j = 0; j < VEC; ++j) sum[j] = stack[level][j] + sum[j];
        if (level < 5)
#pragma unroll
            for (int j = 0; j < VEC; ++j) stack[level][j] = sum[j];
    }
    float* out = a.s1 + row * W + t0;
    if constexpr (VEC == 4) *reinterpret_cast<float4*>(out) = make_float4(sum[0], sum[1], sum[2], sum[3]);
    else *reinterpret_cast<float2*>(out) = make_float2(sum[0], sum[1]);
}

// ZR: the zero-rate rule (Thm. 3) is on; a separate instantiation keeps the plain coder's loop free of it.
// FLEX: the call exports intermediate values or statistics, or uses a per-position step; the plain
// instantiation carries none of those branches in its position loop.
template <int D, int SRC, bool ZR, bool FLEX, int WARPS = kWarpsPerBlock, int BLOCKS = kBlocksPerSM>
__global__ void __launch_bounds__(32 * WARPS, BLOCKS) encode_kernel(const CodecArgs a) {
    constexpr int G = Geo<D>::G;
    constexpr bool FROM_OPEN = SRC == kSrcOpen;
    constexpr bool DENSE = SRC == kSrcDense;
    __shared__ EncTables tb;
    if (FROM_OPEN) chain_next();                             // an append step's first launch may follow
    load_tables(&tb, &a.tables->enc);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const LaneCode lc = lane_code(lane);
    const long long gw = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    uint16_t* stage = a.staging + gw * a.staging_words_per_warp;
    const int cap_words = (int)a.staging_words_per_warp;
    const int Wt = 2 * a.sh.L * a.sh.H, H = a.sh.H, Kp = a.sh.Kp;
    int2* sp0 = g_pair_smem + (threadIdx.x >> 5) * 2 * Kp;
    const int Wl = DENSE ? a.dense_nt : Wt;                  // tables this launch covers
    const unsigned total = FROM_OPEN ? a.open_items : (unsigned)Wl * a.S * a.chunks;
    if (!FROM_OPEN) clear_unused_slots(a, DENSE ? a.dense_t0 : 0, Wl);
    const float inv_d = 1.0f / D, inv_delta = a.sh.inv_delta, inv_delta2 = a.sh.inv_delta2,
                floor2 = a.sh.sigma_floor * a.sh.sigma_floor;
    const int c0 = first_comp<D>(lane);

    constexpr bool QUEUED = SRC == kSrcGather;
    QueueCursor qc = QUEUED ? queue_of_this_sm(a) : QueueCursor{0, 0};
    const unsigned per_table = (unsigned)a.S * (unsigned)a.chunks;
    auto next = [&]() { return QUEUED ? next_queued(a, qc, per_table, Wl, lane) : next_ticket(a.ticket, lane); };
    for (unsigned item = next(); item < total; item = next()) {
        Item it;
        if (FROM_OPEN) {
            const unsigned oi = a.open_first + item;
            it.t = (int)(oi / a.S); it.s = (int)(oi % a.S); it.c = a.chunk_index;
            it.p0 = 0; it.P = a.open_count;
            it.slot = ((long long)it.s * Wt + it.t) * a.st.max_chunks + it.c;
        } else {
            it = bulk_item(a, item, DENSE ? a.dense_t0 : 0);
        }
        if (it.P <= 0) {
            if (lane == 0 && !FROM_OPEN) { a.st.chunk_offset[it.slot] = 0; a.st.chunk_bytes[it.slot] = 0; }
            continue;
        }
        const char* col = reinterpret_cast<const char*>(a.T + (size_t)it.t * a.sh.V * D);
        const float* n2 = a.rownorm2 + (size_t)it.t * a.sh.V;
        uint32_t x = kRansL;
        int wp = cap_words;
        unsigned n_escapes = 0;
        int n_skipped = 0;
        float ideal = 0.f;                                                         // this lane's share, if asked for
        const int2* gp = nullptr;
        const __half* kvp = nullptr;
        const float* s1_at = nullptr;
        int buf = 0;
        if (!FROM_OPEN) {
            if (!DENSE) {
                const long long row = (long long)it.s * a.n + it.p0 + it.P - 1;  // last position first
                gp = a.pairs + row * Kp;
                if (a.s1) s1_at = a.s1 + row * Wt + it.t;
                __syncwarp();                                                    // slot 0 is free again
                prefetch_pairs(sp0, gp, Kp, lane);
            }
            kvp = reinterpret_cast<const __half*>(a.kv.base) + kv_elem(a.kv, it.t, H, it.s, it.p0 + it.P - 1) + c0;
        }
        // dense source: the prediction of the next position is fetched while this one is coded
        float m_next[G] = {};
        float s1_next = 0.f;
        if (DENSE) dense_fetch<D>(a, (long long)it.s * a.n + it.p0 + it.P - 1, it.t - a.dense_t0, c0, m_next, s1_next);
        for (int p = it.P - 1; p >= 0; --p) {
            int sym[G];
            int q;
            bool skip;                                                             // zero-rate position (Thm. 3)
            if (FROM_OPEN) {
                const long long o = ((long long)it.s * Wt + it.t) * a.sh.chunk_pos + p;
                q = a.open_q[o];
                skip = ZR && q <= a.sh.zero_q;
#pragma unroll
                for (int g = 0; g < G; ++g) sym[g] = a.open_sym[o * D + c0 + g];
            } else {
                float mu[G], sigma2;
                uint32_t kv_raw[(G + 1) / 2];
                load_half_raw<G>(kvp, kv_raw);                                     // in flight during the prediction
                kvp -= a.kv.sp;
                if (DENSE) {
                    float m_cur[G];
#pragma unroll
                    for (int g = 0; g < G; ++g) m_cur[g] = m_next[g];
                    const float s1_cur = s1_next;
                    if (p > 0) dense_fetch<D>(a, (long long)it.s * a.n + it.p0 + p - 1, it.t - a.dense_t0, c0, m_next, s1_next);
                    dense_finish<D>(a, it.t - a.dense_t0, c0, inv_d, m_cur, s1_cur, mu, sigma2);
                } else {
                    const int2* sp = sp0 + buf * Kp;
                    if (p > 0) {                                                  // one position ahead
                        gp -= Kp;
                        prefetch_pairs(sp0 + (buf ^ 1) * Kp, gp, Kp, lane);
                        pairs_ready<1>();
                    } else {
                        pairs_ready<0>();
                    }
                    buf ^= 1;
                    predict<D>(col, n2, s1_at, a.pair_index, sp, Kp, lane, inv_d, mu, sigma2);
                    if (s1_at) s1_at -= Wt;
                }
                float inv_delta_p = inv_delta, inv_delta2_p = inv_delta2;
                int zero_q = ZR ? a.sh.zero_q : 0;
                if (FLEX && a.step_exp) {                                          // adaptive step delta * 2^e
                    const int e = a.step_exp[(long long)it.s * a.n + it.p0 + p];
                    inv_delta_p = ldexpf(inv_delta, -e);
                    inv_delta2_p = ldexpf(inv_delta2, -2 * e);
                    if (ZR) zero_q -= 8 * e;                                       // same D against a step 2^e times larger
                }
                q = __reduce_max_sync(kFull, scale_class(sigma2, floor2, inv_delta2_p));   // same in all lanes
                skip = ZR && q <= zero_q;
                float kvv[G];
                half_raw_to_float<G>(kv_raw, kvv);
#pragma unroll
                for (int g = 0; g < G; ++g) sym[g] = quantise(kvv[g], mu[g], inv_delta_p);
                __syncwarp();                                                     // readers of this slot are done
                if (FLEX && (a.dbg.sym || a.dbg.q || a.dbg.mu)) {
                    const long long o = ((long long)it.s * a.n + it.p0 + p) * Wt + it.t;
                    if (a.dbg.q && lane == 0) a.dbg.q[o] = q;
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        if (a.dbg.sym) a.dbg.sym[o * D + c0 + g] = skip ? 0 : sym[g];
                        if (a.dbg.mu) a.dbg.mu[o * D + c0 + g] = mu[g];
                    }
                }
            }
            if (ZR && skip) { ++n_skipped; continue; }                             // nothing is coded
            int s, qp;
            class_params(q, s, qp);
            if (FLEX && a.dbg.ideal) {              // statistics only: log2(2^15 / f) + s raw bits (+ 32 per escape)
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const uint32_t at = (uint32_t)(((sym[g] + (s ? (1 << (s - 1)) : 0)) >> s) + kHiMax);
                    const uint32_t f = tb.enc[qp - kQMin][min(at, (uint32_t)kEsc)].fc & 0xffffu;
                    ideal += (float)(kProbBits + s) - log2f((float)f) + (at > 2u * kHiMax ? 32.f : 0.f);
                }
            }
            wp = encode_position<G>(sym, s, tb.enc[qp - kQMin], x, stage, wp, lc, n_escapes);
        }
        if (FLEX && a.dbg.ideal) {
            ideal = warp_sum(ideal);
            if (lane == 0) atomicAdd(&a.counters->ideal_bits, (double)ideal);
        }
        commit_chunk(a, it.slot, x, stage, wp, cap_words, lane, it.P, n_escapes, n_skipped);
        __syncwarp();
    }
}

template <int D, bool DENSE, bool ZR, bool FLEX, int WARPS = kWarpsPerBlock, int BLOCKS = kBlocksPerSM>
__global__ void __launch_bounds__(32 * WARPS, BLOCKS) decode_kernel(const CodecArgs a) {
    constexpr int G = Geo<D>::G;
    __shared__ DecTables tb;
    load_tables(&tb, &a.tables->dec);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const LaneCode lc = lane_code(lane);
    const int Wt = 2 * a.sh.L * a.sh.H, H = a.sh.H, Kp = a.sh.Kp;
    int2* sp0 = g_pair_smem + (threadIdx.x >> 5) * 2 * Kp;
    const int Wl = DENSE ? a.dense_nt : Wt;
    const unsigned total = (unsigned)Wl * a.S * a.chunks;
    const float inv_d = 1.0f / D, delta = a.sh.delta, inv_delta2 = a.sh.inv_delta2,
                floor2 = a.sh.sigma_floor * a.sh.sigma_floor;
    const int c0 = first_comp<D>(lane);

    QueueCursor qc = DENSE ? QueueCursor{0, 0} : queue_of_this_sm(a);
    const unsigned per_table = (unsigned)a.S * (unsigned)a.chunks;
    auto next = [&]() { return DENSE ? next_ticket(a.ticket, lane) : next_queued(a, qc, per_table, Wl, lane); };
    for (unsigned item = next(); item < total; item = next()) {
        const Item it = bulk_item(a, item, DENSE ? a.dense_t0 : 0);
        if (it.P <= 0) continue;
        const unsigned long long off = a.st.chunk_offset[it.slot];
        const unsigned nbytes = a.st.chunk_bytes[it.slot];
        if (nbytes < 128u || (nbytes & 1u) || (off & 15ull) || off + nbytes > a.st.capacity) {
            if (lane == 0) atomicOr(a.status, kStCorrupt);
            continue;
        }
        const uint8_t* src = a.st.payload + off;
        uint32_t x = reinterpret_cast<const uint32_t*>(src)[lane];
        bool bad = x < kRansL;
        const uint16_t* words = reinterpret_cast<const uint16_t*>(src + 128);
        const int nwords = (int)((nbytes - 128u) >> 1);
        const int last = nwords - 1;                 // -1 for a chunk of states only: words[-1] is inside the chunk
        auto read_word = [&](int i) { return (uint32_t)__ldg(words + min(i, last)); };   // past the end: the last word
        int rp = 0;
        const char* col = reinterpret_cast<const char*>(a.T + (size_t)it.t * a.sh.V * D);
        const float* n2 = a.rownorm2 + (size_t)it.t * a.sh.V;
        const int2* gp = a.pairs + ((long long)it.s * a.n + it.p0) * Kp;
        const float* s1_at = !DENSE && a.s1 ? a.s1 + ((long long)it.s * a.n + it.p0) * Wt + it.t : nullptr;
        __syncwarp();
        if (!DENSE) prefetch_pairs(sp0, gp, Kp, lane);
        int buf = 0;
        long long kvo = kv_elem(a.kv, it.t, H, it.s, it.p0) + c0;
        float m_next[G] = {};
        float s1_next = 0.f;
        if (DENSE) dense_fetch<D>(a, (long long)it.s * a.n + it.p0, it.t - a.dense_t0, c0, m_next, s1_next);
        for (int p = 0; p < it.P; ++p) {
            float mu[G], sigma2;
            if (DENSE) {
                float m_cur[G];
#pragma unroll
                for (int g = 0; g < G; ++g) m_cur[g] = m_next[g];
                const float s1_cur = s1_next;
                if (p + 1 < it.P) dense_fetch<D>(a, (long long)it.s * a.n + it.p0 + p + 1, it.t - a.dense_t0, c0, m_next, s1_next);
                dense_finish<D>(a, it.t - a.dense_t0, c0, inv_d, m_cur, s1_cur, mu, sigma2);
            } else {
                const int2* sp = sp0 + buf * Kp;
                if (p + 1 < it.P) {
                    gp += Kp;
                    prefetch_pairs(sp0 + (buf ^ 1) * Kp, gp, Kp, lane);
                    pairs_ready<1>();
                } else {
                    pairs_ready<0>();
                }
                buf ^= 1;
                predict<D>(col, n2, s1_at, a.pair_index, sp, Kp, lane, inv_d, mu, sigma2);
                if (s1_at) s1_at += Wt;
            }
            float delta_p = delta, inv_delta2_p = inv_delta2;
            int zero_q = ZR ? a.sh.zero_q : 0;
            if (FLEX && a.step_exp) {
                const int e = a.step_exp[(long long)it.s * a.n + it.p0 + p];
                delta_p = ldexpf(delta, e);
                inv_delta2_p = ldexpf(inv_delta2, -2 * e);
                if (ZR) zero_q -= 8 * e;
            }
            const int q = __reduce_max_sync(kFull, scale_class(sigma2, floor2, inv_delta2_p));   // same in all lanes
            __syncwarp();                                                         // readers of this slot are done
            int sym[G];
            float out[G];
            if (ZR && q <= zero_q) {                                              // zero-rate position: KV' = KV^
#pragma unroll
                for (int g = 0; g < G; ++g) { sym[g] = 0; out[g] = mu[g]; }
            } else {
                int s, qp;
                class_params(q, s, qp);
                decode_position<G>(sym, s, Lookup{tb.first[qp - kQMin], tb.fc[qp - kQMin]}, x, read_word, rp, lc);
#pragma unroll
                for (int g = 0; g < G; ++g) out[g] = __fmaf_rn((float)sym[g], delta_p, mu[g]);
            }
            store_vec<G>(a.kv.base, kvo, out, a.sh.out_dtype);
            kvo += a.kv.sp;
            if (FLEX && (a.dbg.sym || a.dbg.q || a.dbg.mu)) {
                const long long o = ((long long)it.s * a.n + it.p0 + p) * Wt + it.t;
                if (a.dbg.q && lane == 0) a.dbg.q[o] = q;
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    if (a.dbg.sym) a.dbg.sym[o * D + c0 + g] = sym[g];
                    if (a.dbg.mu) a.dbg.mu[o * D + c0 + g] = mu[g];
                }
            }
        }
        bad = bad || x != kRansL || rp != nwords;
        if (__any_sync(kFull, bad) && lane == 0) atomicOr(a.status, kStCorrupt);
    }
}

// In-place orthonormal Walsh-Hadamard transform of a d-vector spread over the warp in the coder's
// ownership (lane l, register g  <->  component 8 (l mod R) + G (l div R) + g): every bit of the
// component index is either a bit of g (butterflies between registers) or a bit of the lane number
// (butterflies by shuffle), so log2(G) + 5 = log2(d) stages visit every bit once; the element whose
// bit is set receives partner - self.  Output index = input index (natural Hadamard order).
template <int D>
__device__ __forceinline__ void hadamard(float (&v)[Geo<D>::G], int lane) {
    constexpr int G = Geo<D>::G;
#pragma unroll
    for (int m = 1; m < G; m <<= 1) {
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (!(g & m)) { const float a = v[g], b = v[g | m]; v[g] = a + b; v[g | m] = a - b; }
    }
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
        const bool up = (lane & m) != 0;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const float p = __shfl_xor_sync(kFull, v[g], m);
            v[g] = up ? p - v[g] : v[g] + p;
        }
    }
    constexpr float norm = D == 32 ? 0.17677669529663687f : D == 64 ? 0.125f : D == 128 ? 0.08838834764831845f : 0.0625f;   // d^(-1/2)
#pragma unroll
    for (int g = 0; g < G; ++g) v[g] *= norm;
}

template <int D, bool WIDEN>
constexpr int kRotqBlocks = WIDEN && D != 256 ? 3 : kGatherBlocks;       // an SM; see launch_rotq
// Rotated fixed-rate quantiser (Prop. 3 step 3: a per-vector quantiser on the residual R = KV - KV^):
// x = eps * R, y = H x (orthonormal Hadamard), s = max |y|, b-bit mid-rise codes on [-s, s]; the
// record is s followed by one ballot word per (register, code bit).  ENC: KV -> records;
// otherwise records -> KV' = KV^ + eps * H y^.  One warp per (stream, chunk of positions).
template <int D, bool ENC, bool WIDEN>
__global__ void __launch_bounds__(kThreads, (kRotqBlocks<D, WIDEN>)) rotq_kernel(const CodecArgs a, const RotqArgs rq) {
    constexpr int G = Geo<D>::G;
    const int lane = threadIdx.x & 31;
    const int Wt = 2 * a.sh.L * a.sh.H, H = a.sh.H, Kp = a.sh.Kp, B = rq.bits;
    int2* sp0 = g_pair_smem + (threadIdx.x >> 5) * 2 * Kp;
    const unsigned total = (unsigned)Wt * a.S * a.chunks;
    const float inv_d = 1.0f / D, half_levels = 0.5f * (float)(1 << B), cell = 2.0f / (float)(1 << B);
    const int c0 = first_comp<D>(lane);
    float sgn[G];
#pragma unroll
    for (int g = 0; g < G; ++g) sgn[g] = (rq.sign_bits[(c0 + g) >> 5] >> ((c0 + g) & 31)) & 1u ? -1.0f : 1.0f;
    QueueCursor qc = queue_of_this_sm(a);
    const unsigned per_table = (unsigned)a.S * (unsigned)a.chunks;
    for (unsigned item = next_queued(a, qc, per_table, Wt, lane); item < total; item = next_queued(a, qc, per_table, Wt, lane)) {
        const Item it = bulk_item(a, item);
        if (it.P <= 0) continue;
        const char* col = reinterpret_cast<const char*>(a.T + (size_t)it.t * a.sh.V * D);
        const float* n2 = a.rownorm2 + (size_t)it.t * a.sh.V;
        const int2* gp = a.pairs + ((long long)it.s * a.n + it.p0) * Kp;
        __syncwarp();
        prefetch_pairs(sp0, gp, Kp, lane);
        int buf = 0;
        long long kvo = kv_elem(a.kv, it.t, H, it.s, it.p0) + c0;
        uint32_t* rec = rq.records + (((long long)it.s * Wt + it.t) * a.n + it.p0) * rq.rec_words;
        for (int p = 0; p < it.P; ++p, rec += rq.rec_words, kvo += a.kv.sp) {
            const int2* sp = sp0 + buf * Kp;
            if (p + 1 < it.P) {
                gp += Kp;
                prefetch_pairs(sp0 + (buf ^ 1) * Kp, gp, Kp, lane);
                pairs_ready<1>();
            } else {
                pairs_ready<0>();
            }
            buf ^= 1;
            float mu[G], sigma2;
            predict<D, WIDEN, WIDEN, true>(col, n2, nullptr, a.pair_index, sp, Kp, lane, inv_d, mu, sigma2);
            __syncwarp();                                                         // readers of this slot are done
            float y[G];
            if (ENC) {
                load_half_vec<G>(reinterpret_cast<const __half*>(a.kv.base) + kvo, y);
#pragma unroll
                for (int g = 0; g < G; ++g) y[g] = __fsub_rn(y[g], mu[g]) * sgn[g];
                hadamard<D>(y, lane);
                float amax = 0.f;
#pragma unroll
                for (int g = 0; g < G; ++g) amax = fmaxf(amax, fabsf(y[g]));
                const float scale = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(amax)));   // non-negative floats order like their bits
                const float inv = scale > 0.f ? __fdiv_rn(1.0f, scale) : 0.f;
                uint32_t mine0 = __float_as_uint(scale), mine1 = 0u;               // word 0 of the record is the scale
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    int c = (int)floorf(__fmaf_rn(__fmul_rn(y[g], inv), half_levels, half_levels));
                    c = min(max(c, 0), (1 << B) - 1);
                    for (int b = 0; b < B; ++b) {
                        const uint32_t plane = __ballot_sync(kFull, (c >> b) & 1);
                        const int w = 1 + g * B + b;
                        if ((w & 31) == lane) { if (w < 32) mine0 = plane; else mine1 = plane; }
                    }
                }
                if (lane < rq.rec_words) rec[lane] = mine0;                         // rec_words <= 64
                if (lane + 32 < rq.rec_words) rec[lane + 32] = mine1;
            } else {
                const uint32_t w0 = lane < rq.rec_words ? __ldg(rec + lane) : 0u;
                const uint32_t w1 = lane + 32 < rq.rec_words ? __ldg(rec + lane + 32) : 0u;
                const float scale = __uint_as_float(__shfl_sync(kFull, w0, 0));
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    int c = 0;
                    for (int b = 0; b < B; ++b) {
                        const int w = 1 + g * B + b;
                        const uint32_t plane = __shfl_sync(kFull, w < 32 ? w0 : w1, w & 31);
                        c |= (int)((plane >> lane) & 1u) << b;
                    }
                    y[g] = scale * __fmaf_rn((float)c + 0.5f, cell, -1.0f);
                }
                hadamard<D>(y, lane);
                float out[G];
#pragma unroll
                for (int g = 0; g < G; ++g) out[g] = __fadd_rn(mu[g], y[g] * sgn[g]);
                store_vec<G>(a.kv.base, kvo, out, a.sh.out_dtype);
            }
        }
    }
}

// Decode-time append: one warp per (session, table) predicts the new position and stores its
// symbols and class in slot a.open_slot of the stream's open chunk.  The rows come from HBM at
// random, so what counts is row loads in flight: four blocks per SM (64 registers, the whole
// unrolled batch of row loads issued before the first use) measured best.
template <int D>
__global__ void __launch_bounds__(kThreads, kGatherBlocks) append_quantise_kernel(const CodecArgs a) {
    constexpr int G = Geo<D>::G;
    chain_next();
    chain_wait();
    const int lane = threadIdx.x & 31;
    const int Wt = 2 * a.sh.L * a.sh.H, H = a.sh.H, Kp = a.sh.Kp;
    int2* sp = g_pair_smem + (threadIdx.x >> 5) * 2 * Kp;
    const long long gw = (long long)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    const long long nw = (long long)gridDim.x * kWarpsPerBlock;
    const float inv_d = 1.0f / D, inv_delta = a.sh.inv_delta, inv_delta2 = a.sh.inv_delta2,
                floor2 = a.sh.sigma_floor * a.sh.sigma_floor;
    const int c0 = first_comp<D>(lane);
    for (long long item = gw; item < (long long)Wt * a.S; item += nw) {
        const int t = (int)from_lane0((unsigned)(item / a.S), lane), b = (int)(item % a.S);
        const char* col = reinterpret_cast<const char*>(a.T + (size_t)t * a.sh.V * D);
        const int2* gp = a.pairs + (long long)b * Kp;
        __syncwarp();
        prefetch_pairs(sp, gp, Kp, lane);
        pairs_ready<0>();
        float kvv[G];
        load_half_vec<G>(reinterpret_cast<const __half*>(a.kv.base) + kv_elem(a.kv, t, H, b, 0) + c0, kvv);
        float mu[G], sigma2;
        predict<D>(col, a.rownorm2 + (size_t)t * a.sh.V, nullptr, a.pair_index, sp, Kp, lane, inv_d, mu, sigma2);
        const int q = scale_class(sigma2, floor2, inv_delta2);
        const long long o = ((long long)b * Wt + t) * a.sh.chunk_pos + a.open_slot;
        if (lane == 0) a.open_q[o] = q;
#pragma unroll
        for (int g = 0; g < G; ++g) a.open_sym[o * D + c0 + g] = q <= a.sh.zero_q ? 0 : quantise(kvv[g], mu[g], inv_delta);
    }
}

// Dynamic shared memory of the kernels that stage pairs: one slot of Kp entries per warp.
template <class Kern>
cudaError_t pair_smem_bytes(Kern kern, int Kp, size_t& bytes) {
    bytes = (size_t)kWarpsPerBlock * 2 * Kp * sizeof(int2);
    return bytes > 24 * 1024 ? allow_smem(kern, bytes) : cudaSuccess;
}

// Gather kernels with a coder: one block an SM; where the pairs of that many warps do not fit beside each
// other (K above 320, above 426 with 24 warps), blocks of eight, as many as fit.
template <class Kern>
cudaError_t launch_gather(const CodecArgs& a, Kern kern, int warps, cudaStream_t st) {
    int blocks = sm_count();
    size_t bytes = (size_t)warps * 2 * a.sh.Kp * sizeof(int2);
    if (bytes > kMostSmem) { blocks *= warps / kWarpsPerBlock; bytes /= warps / kWarpsPerBlock; warps = kWarpsPerBlock; }
    const cudaError_t e = allow_smem(kern, bytes);
    if (e != cudaSuccess) return e;
    count_launch();
    return launch_kernel(kern, blocks, 32 * warps, bytes, st, false, 1, a);
}

}  // namespace

int codec_grid_warps(int) { return sm_count() * kBlocksPerSM * kWarpsPerBlock; }

// Chunks an SM is counted to take from a queue, as when five blocks were resident on one.  32, the warps that
// are now, gives fewer and wider queues (19 of 8 SMs instead of 25 of 6 for 256 chunks a table): 64 uniform rows a
// vector from HBM, encode, 2.57 -> 2.38 ns a vector with all chunks full, 2.69 -> 2.68 with ragged sessions, skewed
// rows equal; it would change the layout that plc_last_schedule reports, so 40 stays.
constexpr int kQueueItems = 40;
static_assert(kQueueItems >= kGatherBlocks * kWarpsPerBlock, "a queue must keep its SMs busy");
static void set_queues(CodecArgs& a, int n_tables, int items_per_sm = kQueueItems);

// A block per chunk (plc_coop.cu) while the chunks would not fill the GPU with a warp each: below that a
// warp's own chain is what the call waits for; above it the kernels here do more work per instruction
// (65536 chunks: 12.6 ms a layer group against 11.3).
static bool use_coop(const CodecArgs& a) {
    const long long items = (long long)(a.mu_dense ? a.dense_nt : 2 * a.sh.L * a.sh.H) * a.S * a.chunks;
    return items <= (long long)sm_count() * kWarpsPerBlock * (a.mu_dense ? kBlocksPerSM : kGatherBlocks);
}
constexpr int kCoopItems = 4;                    // chunks an SM works on at a time there

// Queue layout of a gather launch.  With one queue for the whole GPU the resident warps span
// about (resident warps / chunks per table) + 1 consecutive tables; if those tables fit in L2 that
// is the layout with the smallest working set and it is kept.  Otherwise L2 cannot hold the tables
// in flight whatever the order, and the only reuse left is between positions that share candidate
// rows: then a queue is served by as few SMs as keep busy with ONE table's chunks (rounded down),
// so that the warps of an SM gather from one or two tables and shared rows stay in that SM's L1.
void codec_schedule(const CodecArgs& a0, int n_tables, int* nq, int* g) {
    CodecArgs a = a0;
    set_queues(a, n_tables, use_coop(a) ? kCoopItems : kQueueItems);
    *nq = a.sched_nq; *g = a.sched_g;
}

static void set_queues(CodecArgs& a, int n_tables, int items_per_sm) {
    const int sms = sm_count(), warps_per_sm = items_per_sm;
    const long long per_table = std::max(1LL, (long long)a.S * a.chunks);
    const long long spanned = ((long long)sms * warps_per_sm + per_table - 1) / per_table + 1;
    const double table_bytes = 2.0 * a.sh.V * a.sh.d;
    int dev = 0, l2 = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
    long long g = per_table / warps_per_sm;
    if ((double)std::min<long long>(spanned, n_tables) * table_bytes <= (double)l2) g = sms;
    g = std::max(1LL, std::min<long long>(g, sms));
    int nq = (sms + (int)g - 1) / (int)g;
    nq = std::max(1, std::min(nq, std::min(n_tables, kTicketWords)));
    a.sched_g = (int)g; a.sched_nq = nq;
}

cudaError_t launch_rownorm(const __half* T, float* out, long long rows, int d, unsigned int* not_finite, cudaStream_t st) {
    return dispatch_d(d, [&](auto D) {
        constexpr int a_block = 8 * kNormRows;
        const long long blocks = std::min((rows + a_block - 1) / a_block, (long long)sm_count() * 16);
        rownorm_kernel<decltype(D)::value><<<(unsigned)blocks, 256, 0, st>>>(T, out, rows, not_finite);
        count_launch();
        return cudaGetLastError();
    });
}

cudaError_t launch_norms_by_row(const float* norms, float* by_row, int V, int tables, cudaStream_t st) {
    norms_by_row_kernel<<<dim3((unsigned)((V + 31) / 32), (unsigned)((tables + 31) / 32)), 256, 0, st>>>(norms, by_row, V, tables);
    count_launch();
    return cudaGetLastError();
}

static int log2_of(int v) { return v > 1 ? 1 + log2_of(v >> 1) : 0; }

cudaError_t launch_variance(const CodecArgs& a, cudaStream_t st) {
    const int W = 2 * a.sh.L * a.sh.H, vec = W % 4 == 0 ? 4 : 2;
    int width = 1;
    while (width < 32 && width * vec < W) width *= 2;
    const long long rows = (long long)a.S * a.n, a_block = 8 * (32 / width);
    auto kern = vec == 4 ? variance_kernel<4> : variance_kernel<2>;
    kern<<<dim3((unsigned)((rows + a_block - 1) / a_block), (unsigned)((W + width * vec - 1) / (width * vec))), 256, 0, st>>>(a, width, a.pair_index ? 0 : log2_of(2 * a.sh.d), log2_of(256 / a.sh.d));
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_encode(const CodecArgs& a0, cudaStream_t st) {
    CodecArgs a = a0;
    const int items_per_sm = use_coop(a) ? kCoopItems : kQueueItems;
    set_queues(a, 2 * a.sh.L * a.sh.H, items_per_sm);
    if (a.mu_dense) {
        const cudaError_t e = cudaMemsetAsync(a.ticket, 0, sizeof(unsigned int), st);
        if (e != cudaSuccess) return e;
    }
    if (use_coop(a)) return launch_coop(a, true, st);
    const bool zr = a.sh.zero_q != kZeroOff;
    const bool flex = a.dbg.sym || a.dbg.q || a.dbg.mu || a.dbg.ideal || a.step_exp;
    return dispatch_d(a.sh.d, [&](auto D) {
        constexpr int d = decltype(D)::value;
        if (a.mu_dense) {
            auto kd = zr ? (flex ? encode_kernel<d, kSrcDense, true, true> : encode_kernel<d, kSrcDense, true, false>)
                         : (flex ? encode_kernel<d, kSrcDense, false, true> : encode_kernel<d, kSrcDense, false, false>);
            kd<<<sm_count() * kBlocksPerSM, kThreads, 0, st>>>(a);
            count_launch();
            return cudaGetLastError();
        }
        auto pick = [&](auto warps) {
            constexpr int N = decltype(warps)::value;
            return zr ? (flex ? encode_kernel<d, kSrcGather, true, true, N, 1> : encode_kernel<d, kSrcGather, true, false, N, 1>)
                      : (flex ? encode_kernel<d, kSrcGather, false, true, N, 1> : encode_kernel<d, kSrcGather, false, false, N, 1>);
        };
        return a.sched_nq == 1 ? launch_gather(a, pick(std::integral_constant<int, kFarWarps>{}), kFarWarps, st)
                               : launch_gather(a, pick(std::integral_constant<int, kGatherWarps>{}), kGatherWarps, st);
    });
}

cudaError_t launch_append_seal(const CodecArgs& a, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(a.ticket, 0, sizeof(unsigned int), st);
    if (e != cudaSuccess) return e;
    return dispatch_d(a.sh.d, [&](auto D) {
        long long warps = (long long)a.open_items;
        long long blocks = (warps + kWarpsPerBlock - 1) / kWarpsPerBlock;
        if (blocks > (long long)sm_count() * kBlocksPerSM) blocks = (long long)sm_count() * kBlocksPerSM;
        auto ko = a.sh.zero_q != kZeroOff ? encode_kernel<decltype(D)::value, kSrcOpen, true, false> : encode_kernel<decltype(D)::value, kSrcOpen, false, false>;
        ko<<<(unsigned)blocks, kThreads, 0, st>>>(a);
        count_launch();
        return cudaGetLastError();
    });
}

cudaError_t launch_decode(const CodecArgs& a0, cudaStream_t st) {
    CodecArgs a = a0;
    const int items_per_sm = use_coop(a) ? kCoopItems : kQueueItems;
    set_queues(a, 2 * a.sh.L * a.sh.H, items_per_sm);
    if (a.mu_dense) {
        const cudaError_t e = cudaMemsetAsync(a.ticket, 0, sizeof(unsigned int), st);
        if (e != cudaSuccess) return e;
    }
    if (use_coop(a)) return launch_coop(a, false, st);
    const bool zr = a.sh.zero_q != kZeroOff;
    const bool flex = a.dbg.sym || a.dbg.q || a.dbg.mu || a.step_exp;
    return dispatch_d(a.sh.d, [&](auto D) {
        constexpr int d = decltype(D)::value;
        if (a.mu_dense) {
            auto kd = zr ? (flex ? decode_kernel<d, true, true, true> : decode_kernel<d, true, true, false>)
                         : (flex ? decode_kernel<d, true, false, true> : decode_kernel<d, true, false, false>);
            kd<<<sm_count() * kBlocksPerSM, kThreads, 0, st>>>(a);
            count_launch();
            return cudaGetLastError();
        }
        auto pick = [&](auto warps) {
            constexpr int N = decltype(warps)::value;
            return zr ? (flex ? decode_kernel<d, false, true, true, N, 1> : decode_kernel<d, false, true, false, N, 1>)
                      : (flex ? decode_kernel<d, false, false, true, N, 1> : decode_kernel<d, false, false, false, N, 1>);
        };
        return a.sched_nq == 1 ? launch_gather(a, pick(std::integral_constant<int, kFarWarps>{}), kFarWarps, st)
                               : launch_gather(a, pick(std::integral_constant<int, kGatherWarps>{}), kGatherWarps, st);
    });
}

// Rows are widened on the tensor cores where a queue is served by a few SMs (set_queues: the tables in flight are more
// than L2 holds), with 24 warps an SM at 80 registers (32 at 64 for 256 components); where all SMs share a queue, and for
// T that the tensor cores cannot take, value by value with 32 warps.  4000 positions, 8 x 8 heads of 128, K = 64, both calls, value by value with stretches of 32 rows / widened
// with 32 warps / as now, us: V = 32000, skewed candidates (many queues) 1693 / 1457 / 1433, uniform 2742 / 3103 / 2616,
// uniform K = 128 4925 / 5802 / 4720; V = 5000 (one queue) 1360 / 1480 / 1319; 4 layers (one queue) skewed 834 / 854 /
// 814, uniform 1055 / 1290 / 996; 256 components, 4 layers, skewed 1648 / 1398 / 1355 (24 warps 1387), uniform 2725 /
// 2744 / 2740 (3000).
cudaError_t launch_rotq(const CodecArgs& a0, const RotqArgs& r, bool encode, cudaStream_t st) {
    CodecArgs a = a0;
    set_queues(a, 2 * a.sh.L * a.sh.H);
    const bool widen = a.sched_nq > 1 && a.finite && !a.pair_index;
    return dispatch_d(a.sh.d, [&](auto D) {
        constexpr int d = decltype(D)::value;
        auto kern = widen ? (encode ? rotq_kernel<d, true, true> : rotq_kernel<d, false, true>)
                          : (encode ? rotq_kernel<d, true, false> : rotq_kernel<d, false, false>);
        size_t sm = 0;
        cudaError_t e2 = pair_smem_bytes(kern, a.sh.Kp, sm);
        if (e2 != cudaSuccess) return e2;
        count_launch();
        return launch_kernel(kern, sm_count() * (widen ? kRotqBlocks<d, true> : kRotqBlocks<d, false>), kThreads, sm, st, false, 1, a, r);
    });
}

cudaError_t launch_append_quantise(const CodecArgs& a, cudaStream_t st) {
    return dispatch_d(a.sh.d, [&](auto D) {
        long long warps = (long long)a.S * 2 * a.sh.L * a.sh.H;
        long long blocks = (warps + kWarpsPerBlock - 1) / kWarpsPerBlock;
        auto kern = append_quantise_kernel<decltype(D)::value>;
        size_t sm = 0;
        cudaError_t e2 = pair_smem_bytes(kern, a.sh.Kp, sm);
        if (e2 != cudaSuccess) return e2;
        // one wave: as many blocks as are resident together, each walking its share of the items
        int occ = 1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kThreads, sm) != cudaSuccess || occ < 1) occ = 1;
        if (blocks > (long long)sm_count() * occ) blocks = (long long)sm_count() * occ;
        count_launch();
        return launch_kernel(kern, (unsigned)blocks, kThreads, sm, st, a.behind > 0, 1, a);
    });
}

}  // namespace plc
