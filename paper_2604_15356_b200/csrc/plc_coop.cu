// Predict / quantise / rANS with a whole block per (stream, chunk), for calls with few chunks.
//
// The kernels of plc_codec.cu give every chunk to one warp, which predicts a position and codes it
// before it turns to the next: right while there are enough chunks to fill the GPU, but a call with
// fewer chunks than resident warps then runs at the latency of one warp's chain (row gathers, the KV
// load, the coder), about 1.8 us a position however little work there is.  Only the coder is serial
// in a chunk, and of the coder only the state and the word cursor; the rest is independent from
// position to position.  Here warp 0 of a block carries the chunk's state and the other warps do
// everything else, one position each and batch, two batches deep in shared memory with one barrier a
// batch: encoding, they predict, quantise, look the table entries up and transpose the bit planes, and a
// batch later put the words where the coder has found their places; decoding, they predict (the coder
// needs the class) and, a batch later, fetch the planes whose places the coder has found and write the
// vectors.  The coder itself is the bottleneck of a block (it never waits at the barrier), and every
// instruction of it counts: 940 cycles a position of 128 components when it also placed the words.
// The decoder's words come through a ring in shared memory filled by asynchronous copies, so no
// refill waits for global memory.
#include <algorithm>

#include "plc_codec.cuh"

namespace plc {
namespace {

// Predicting warps of a block.
__host__ __device__ constexpr int coop_predictors(int warps) { return warps >= 16 ? 3 * warps / 4 : warps - 1; }
constexpr int kRingBlock = 512;                          // bytes one warp-wide copy brings to the word ring of a decoding coder
// Ring size: a position takes at most G * (2 * 15 + 32 + 64) words.  The roomy ring holds two positions at a
// time for the coder (of blocks whose predictions come from memory, or that have an SM to themselves);
// where blocks gather rows beside each other the 4 KB more a block cost more L1 than the coder gains.
__host__ __device__ constexpr int ring_bytes(int G, bool roomy) { return (G == 8 ? 8192 : 4096) * (roomy ? 2 : 1); }

// What a predicting warp tells the coder about a position (one 16-byte word): bit planes (-1: nothing is
// coded), table id - kQMin, whether a component escapes (encoding; decoding: the coder's answer).
struct __align__(16) SlotMeta { int planes, table, escaped, pad; };

// The words of a chunk, read through the ring.  `ready` bytes have landed, `fetched` are on their way.
template <int BYTES>
struct RingWords {
    const uint16_t* ring;
    __device__ __forceinline__ uint32_t operator()(int i) const { return ring[i & (BYTES / 2 - 1)]; }
};
template <int BYTES>
__device__ __forceinline__ void ring_fetch(uint16_t* ring, const uint8_t* src, int total, int rp, int& fetched, int lane) {
    while (fetched < total && fetched + kRingBlock <= 2 * rp + BYTES) {
        const int at = fetched + 16 * lane;
        if (at < total) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(reinterpret_cast<unsigned char*>(ring) + (at & (BYTES - 1)));
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src + at), "r"(min(16, total - at)) : "memory");
        }
        fetched += kRingBlock;
    }
}

// A position's slot.  Encoding: in, the table entries of its steps (u itself where a component escapes);
// out, over them, the state before each step, and behind them the lanes that emit at each step and the
// place of the position's words.  Decoding, out: the steps' symbols (the position's symbols themselves
// where one escapes) and behind them the steps' places in the word stream.
constexpr int kTailWords = 12;                           // 8 words, one a step, and the place; padded to 16 bytes
template <int G>
constexpr int kEncSlotWords = 64 * G + kTailWords;
template <int G>
constexpr int kDecSlotWords = 32 * G + kTailWords;
// v[0 .. G) for all lanes, the same value in every lane.
template <int G, class V>
__device__ __forceinline__ void tail_put(int* tail, const V (&v)[G]) {
    if constexpr (G >= 4) {
#pragma unroll
        for (int i = 0; i < G / 4; ++i) reinterpret_cast<int4*>(tail)[i] = make_int4((int)v[4 * i], (int)v[4 * i + 1], (int)v[4 * i + 2], (int)v[4 * i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < G; ++i) tail[i] = (int)v[i];
    }
}
template <int G, class V>
__device__ __forceinline__ void tail_get(const int* tail, V (&v)[G]) {
#pragma unroll
    for (int i = 0; i < G; ++i) v[i] = (V)tail[i];
}
template <int G>
__device__ __forceinline__ void slot_put_ints(int* slot, int lane, const int (&v)[G]) {
    if constexpr (G >= 4) {
#pragma unroll
        for (int i = 0; i < G / 4; ++i) reinterpret_cast<int4*>(slot)[i * 32 + lane] = make_int4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < G; ++i) slot[i * 32 + lane] = v[i];
    }
}
template <int G>
__device__ __forceinline__ void slot_get_ints(const int* slot, int lane, int (&v)[G]) {
    if constexpr (G >= 4) {
#pragma unroll
        for (int i = 0; i < G / 4; ++i) {
            const int4 w = reinterpret_cast<const int4*>(slot)[i * 32 + lane];
            v[4 * i] = w.x; v[4 * i + 1] = w.y; v[4 * i + 2] = w.z; v[4 * i + 3] = w.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < G; ++i) v[i] = slot[i * 32 + lane];
    }
}
template <int G>
__device__ __forceinline__ void slot_put_entries(int* slot, int lane, const EncEntry (&e)[G]) {
    if constexpr (G >= 2) {
#pragma unroll
        for (int i = 0; i < G / 2; ++i)
            reinterpret_cast<uint4*>(slot)[i * 32 + lane] = make_uint4(e[2 * i].rcp, e[2 * i].fc, e[2 * i + 1].rcp, e[2 * i + 1].fc);
    } else {
        reinterpret_cast<uint2*>(slot)[lane] = make_uint2(e[0].rcp, e[0].fc);
    }
}
template <int G>
__device__ __forceinline__ void slot_get_entries(const int* slot, int lane, EncEntry (&e)[G]) {
    if constexpr (G >= 2) {
#pragma unroll
        for (int i = 0; i < G / 2; ++i) {
            const uint4 w = reinterpret_cast<const uint4*>(slot)[i * 32 + lane];
            e[2 * i] = EncEntry{w.x, w.y}; e[2 * i + 1] = EncEntry{w.z, w.w};
        }
    } else {
        const uint2 w = reinterpret_cast<const uint2*>(slot)[lane];
        e[0] = EncEntry{w.x, w.y};
    }
}

__host__ __device__ constexpr size_t coop_smem(int warps, int Kp, int d, bool dense, bool enc, bool roomy) {
    const int NP = coop_predictors(warps), G = d / 32, slot = (enc ? 64 : 32) * G + kTailWords;
    return (size_t)(dense ? 0 : NP * 2 * Kp * (int)sizeof(int2)) + (size_t)2 * NP * slot * 4 + (enc ? 0 : ring_bytes(G, roomy));
}

// All warps of a chunk meet here, from different places in the code: those of the block, or of a group of GW.
template <int GW>
struct Meet {
    int group;
    __device__ __forceinline__ void operator()() const {
        if constexpr (GW == 0) asm volatile("barrier.sync 1, %0;" ::"r"((unsigned)(32 + 32 * coop_predictors(blockDim.x >> 5))) : "memory");
        else asm volatile("barrier.sync %0, %1;" ::"r"(1 + group), "n"(32 * GW) : "memory");
    }
};

// The block's current chunk.
struct CoopItem {
    Item it;
    long long row0, kv0;                 // first row of the positions; element of the chunk's first vector
    unsigned long long off;              // decoding: the chunk's bytes
    unsigned nbytes;
    int go;                              // 0: nothing to do for this chunk, -1: no chunks left
};
template <int NP>                        // predicting warps at most
struct CoopShared {
    CoopItem item;
    SlotMeta meta[2][NP];
    uint8_t* dst;                        // encoding: where the finished chunk's words go (null: nowhere)
    int wp;
};

// Warp w (of NP) beside the coder: positions w, w + NP, ... in the coder's order, one a batch; the inputs
// of the next are fetched while it works on one.
template <int D, bool DENSE, bool ENC, bool AHEAD, int GW, class Tab, class Shared>
__device__ __forceinline__ void coop_predict(const CodecArgs& a, Shared& sh, const Tab& tb, int2* sp0, int* slots, int w, int NP,
                                             const Meet<GW>& meet, const LaneCode& lc) {
    constexpr int G = Geo<D>::G, SW = ENC ? kEncSlotWords<G> : kDecSlotWords<G>;
    const int lane = lc.lane;
    const int P = sh.item.it.P, Kp = DENSE ? 0 : a.sh.Kp, n_batches = (P + NP - 1) / NP, c0 = first_comp<D>(lane);
    const int t = (int)from_lane0((unsigned)sh.item.it.t, lane), t0 = DENSE ? a.dense_t0 : 0;
    const int first = ENC ? P - 1 : 0, dir = ENC ? -1 : 1;
    const long long row0 = sh.item.row0;
    const char* col = reinterpret_cast<const char*>(a.T + (size_t)t * a.sh.V * D);
    const int Wt = 2 * a.sh.L * a.sh.H;
    const float* n2 = a.rownorm2 + (size_t)t * a.sh.V;
    const bool zr = a.sh.zero_q != kZeroOff;
    int buf = 0;
    float m_next[G] = {}, s1_next = 0.f, ideal = 0.f;
    uint32_t kv_next[(G + 1) / 2] = {};
    // what finishing the position of the batch before takes, once the coder has passed it: encoding, its bit
    // planes; decoding, its prediction and step
    float mu_old[G] = {};
    uint32_t planes_old[kPlaneWords<G>] = {};
    int s_old = -1, e_old = 0;
    bool esc_old = false;
    auto fetch = [&](int k, int into) {
        const int p = first + dir * k;
        if (DENSE) dense_fetch<D>(a, row0 + p, t - t0, c0, m_next, s1_next);
        else prefetch_pairs(sp0 + into * Kp, a.pairs + (row0 + p) * Kp, Kp, lane);
        if (ENC) load_half_raw<G>(reinterpret_cast<const __half*>(a.kv.base) + sh.item.kv0 + c0 + p * a.kv.sp, kv_next);
    };
    auto finish = [&](int b) {                                                 // the position of batch b
        if (b < 0 || b * NP + w >= P) return;
        const int* slot = slots + ((b & 1) * NP + w) * SW;
        if constexpr (ENC) {
            if (s_old < 0 || esc_old) return;                                  // nothing to write, or written by the coder
            int low[G];
            uint32_t lows[G], emask[G];
            bool emit[G];
            slot_get_ints<G>(slot, lane, low);
            tail_get<G>(slot + 64 * G, emask);
#pragma unroll
            for (int g = 0; g < G; ++g) { lows[g] = (uint32_t)low[g]; emit[g] = (emask[g] >> lane) & 1u; }
            place_position<G>(planes_old, lows, emask, emit, s_old, a.staging + (long long)blockIdx.x * a.staging_words_per_warp,
                              slot[64 * G + 8], lc);
        } else {
            const int p = b * NP + w;
            int sym[G];
            float out[G];
            if (s_old < 0) {                                                   // zero-rate position: KV' = KV^
#pragma unroll
                for (int g = 0; g < G; ++g) { sym[g] = 0; out[g] = mu_old[g]; }
            } else {
                int zz[G];
                slot_get_ints<G>(slot, lane, zz);
                if (sh.meta[b & 1][w].escaped) {
#pragma unroll
                    for (int g = 0; g < G; ++g) sym[g] = zz[g];
                } else {
                    int base[G];
                    tail_get<G>(slot + 32 * G, base);
                    const uint16_t* words = reinterpret_cast<const uint16_t*>(a.st.payload + sh.item.off + 128);
                    const int last = (int)((sh.item.nbytes - 128u) >> 1) - 1;  // past the end: the last word
                    join_position<G>(base, zz, s_old, [&](int i) { return (uint32_t)__ldg(words + min(i, last)); }, lc, sym);
                }
                const float delta = a.step_exp ? ldexpf(a.sh.delta, e_old) : a.sh.delta;
#pragma unroll
                for (int g = 0; g < G; ++g) out[g] = __fmaf_rn((float)sym[g], delta, mu_old[g]);
            }
            store_vec<G>(a.kv.base, sh.item.kv0 + c0 + p * a.kv.sp, out, a.sh.out_dtype);
            if (a.dbg.sym) {
                const long long o = (row0 + p) * (2 * a.sh.L * a.sh.H) + t;
#pragma unroll
                for (int g = 0; g < G; ++g) a.dbg.sym[o * D + c0 + g] = sym[g];
            }
        }
    };
    if (w < P) fetch(w, 0);
    for (int b = 0; b < n_batches; ++b) {
        const int k = b * NP + w, p = first + dir * k;
        float mu[G] = {};
        uint32_t planes[kPlaneWords<G>] = {};
        int s = -1, qp = 0, e = 0;
        bool esc = false;
        if (k < P) {
            float sigma2;
            uint32_t kv_raw[(G + 1) / 2];
#pragma unroll
            for (int i = 0; i < (G + 1) / 2; ++i) kv_raw[i] = kv_next[i];
            if (DENSE) {
                float m_cur[G];
#pragma unroll
                for (int g = 0; g < G; ++g) m_cur[g] = m_next[g];
                const float s1_cur = s1_next;
                if (k + NP < P) fetch(k + NP, 0);
                dense_finish<D>(a, t - t0, c0, 1.0f / D, m_cur, s1_cur, mu, sigma2);
            } else {
                const int2* sp = sp0 + buf * Kp;
                if (k + NP < P) { fetch(k + NP, buf ^ 1); pairs_ready<1>(); }
                else pairs_ready<0>();
                buf ^= 1;
                predict<D, false, (AHEAD || D != 256)>(col, n2, AHEAD ? a.s1 + (row0 + p) * Wt + t : nullptr, a.pair_index, sp, Kp, lane, 1.0f / D, mu, sigma2);
            }
            float inv_delta = a.sh.inv_delta, inv_delta2 = a.sh.inv_delta2;
            int zero_q = a.sh.zero_q;
            if (a.step_exp) {                                                  // adaptive step delta * 2^e
                e = a.step_exp[row0 + p];
                inv_delta = ldexpf(inv_delta, -e);
                inv_delta2 = ldexpf(inv_delta2, -2 * e);
                if (zr) zero_q -= 8 * e;
            }
            const int q = __reduce_max_sync(kFull, scale_class(sigma2, a.sh.sigma_floor * a.sh.sigma_floor, inv_delta2));   // same in all lanes
            const bool skip = zr && q <= zero_q;
            class_params(q, s, qp);
            if constexpr (ENC) {
                float kvv[G];
                half_raw_to_float<G>(kv_raw, kvv);
                int sym[G], u[G];
                uint32_t at[G];
#pragma unroll
                for (int g = 0; g < G; ++g) sym[g] = quantise(kvv[g], mu[g], inv_delta);
                int* slot = slots + ((b & 1) * NP + w) * SW;
                if (split_symbols<G>(sym, s, u, at)) {
                    Prepared<G> pr;
                    prepare_position<G>(u, at, s, tb.enc[qp - kQMin], lc, pr);
                    slot_put_entries<G>(slot, lane, pr.e);
#pragma unroll
                    for (int i = 0; i < kPlaneWords<G>; ++i) planes[i] = pr.plane[i];
                } else {
                    esc = true;
                    slot_put_ints<G>(slot, lane, u);
                }
                if (a.dbg.sym) {
                    const long long o = (row0 + p) * (2 * a.sh.L * a.sh.H) + t;
#pragma unroll
                    for (int g = 0; g < G; ++g) a.dbg.sym[o * D + c0 + g] = skip ? 0 : sym[g];
                }
                if (a.dbg.ideal && !skip) {              // log2(2^15 / f) + s raw bits (+ 32 per escape)
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        const uint32_t f = tb.enc[qp - kQMin][min(at[g], (uint32_t)kEsc)].fc & 0xffffu;
                        ideal += (float)(kProbBits + s) - log2f((float)f) + (at[g] > 2u * kHiMax ? 32.f : 0.f);
                    }
                }
            }
            if (a.dbg.q || a.dbg.mu) {
                const long long o = (row0 + p) * (2 * a.sh.L * a.sh.H) + t;
                if (a.dbg.q && lane == 0) a.dbg.q[o] = q;
#pragma unroll
                for (int g = 0; g < G; ++g)
                    if (a.dbg.mu) a.dbg.mu[o * D + c0 + g] = mu[g];
            }
            if (skip) s = -1;
            if (lane == 0) sh.meta[b & 1][w] = SlotMeta{s, qp - kQMin, esc, 0};
            __syncwarp();                                                      // readers of the pair slot are done
        }
        meet();
        finish(b - 1);
#pragma unroll
        for (int g = 0; g < G; ++g) mu_old[g] = mu[g];
#pragma unroll
        for (int i = 0; i < kPlaneWords<G>; ++i) planes_old[i] = planes[i];
        s_old = s; e_old = e; esc_old = esc;
        __syncwarp();                                                          // the slot's readers are done before it is filled again
    }
    meet();
    finish(n_batches - 1);
    if (ENC && a.dbg.ideal) {
        ideal = warp_sum(ideal);
        if (lane == 0) atomicAdd(&a.counters->ideal_bits, (double)ideal);
    }
}

// Coder of the block's chunk, one batch behind the predictions.
template <int D, bool ENC, bool ROOMY, int GW, class Tab, class Shared>
__device__ __forceinline__ void coop_code(const CodecArgs& a, Shared& sh, const Tab& tb, int* slots, uint16_t* ring, int NP, const Meet<GW>& meet,
                                          const LaneCode& lc) {
    constexpr int G = Geo<D>::G, SW = ENC ? kEncSlotWords<G> : kDecSlotWords<G>;
    const int lane = lc.lane;
    const int P = sh.item.it.P, n_batches = (P + NP - 1) / NP;
    constexpr int kRing = ring_bytes(G, ROOMY);
    uint32_t x = kRansL;
    if constexpr (ENC) {
        uint16_t* stage = a.staging + (long long)blockIdx.x * a.staging_words_per_warp;
        const int cap_words = (int)a.staging_words_per_warp;
        int wp = cap_words, n_skipped = 0;
        unsigned n_escapes = 0;
        for (int b = 0; b < n_batches; ++b) {
            meet();                                                   // batch b is there
            const int cnt = min(NP, P - b * NP);
            int* slot = slots + (b & 1) * NP * SW;
            const SlotMeta* meta = sh.meta[b & 1];
            EncEntry next[G];
            slot_get_entries<G>(slot, lane, next);
            int next_planes = meta[0].planes;
            auto code = [&](const EncEntry (&ent)[G], int planes, int* to) {
                uint32_t low[G], emask[G];
                bool emit[G];
                int lows[G];
                chain_position<G>(ent, x, low, emask, emit);
                wp -= words_of<G>(emask, planes);
#pragma unroll
                for (int g = 0; g < G; ++g) lows[g] = (int)low[g];
                slot_put_ints<G>(to, lane, lows);
                tail_put<G>(to + 64 * G, emask);
                to[64 * G + 8] = wp;
            };
            constexpr int kAhead = ROOMY ? 4 : 1;                              // (beside gathering warps the longer code costs more)
            // One vote a batch: without a position that is skipped or escapes the loop has no branches, and the
            // independent work of neighbouring positions fills the gaps of the state's chain.
            if (!__any_sync(kFull, lane < cnt && (meta[lane].planes < 0 || meta[lane].escaped))) {
#pragma unroll kAhead
                for (int j = 0; j < cnt; ++j, slot += SW) {
                    EncEntry ent[G];
#pragma unroll
                    for (int g = 0; g < G; ++g) ent[g] = next[g];
                    const int planes = next_planes, ahead = j + 1 < cnt ? 1 : 0;         // the last one is fetched again
                    slot_get_entries<G>(slot + ahead * SW, lane, next);
                    next_planes = meta[j + ahead].planes;
                    code(ent, planes, slot);
                }
            } else {
#pragma unroll 1
                for (int j = 0; j < cnt; ++j, slot += SW) {
                    const SlotMeta m = meta[j];
                    if (m.planes < 0) { ++n_skipped; continue; }
                    if (!m.escaped) {
                        EncEntry ent[G];
                        slot_get_entries<G>(slot, lane, ent);
                        code(ent, m.planes, slot);
                    } else {
                        int u[G];
                        slot_get_ints<G>(slot, lane, u);
                        wp = encode_position_escapes<G>(u, m.planes, tb.enc[m.table], x, stage, wp, lane, n_escapes);
                    }
                }
            }
        }
        meet();
        uint8_t* dst = reserve_chunk(a, sh.item.it.slot, x, cap_words - wp, lane, P, n_escapes, n_skipped);
        if (lane == 0) { sh.dst = dst; sh.wp = wp; }
    } else {
        const uint8_t* src = a.st.payload + sh.item.off;
        x = reinterpret_cast<const uint32_t*>(src)[lane];
        bool bad = x < kRansL;
        src += 128;
        const int nwords = (int)((sh.item.nbytes - 128u) >> 1);
        int rp = 0, fetched = 0;
        ring_fetch<kRing>(ring, src, 2 * nwords, 0, fetched, lane);
        const RingWords<kRing> words{ring};
        // rp from which on copies in flight are needed, and from which on more are asked for.  A stretch (two
        // positions in a roomy ring, else one) and its last refill window take at most kStretch + 64 bytes;
        // copies are asked for at least every kFetchStep words and a stretch, so at least ring - 512 -
        // 2 kFetchStep - kStretch bytes ahead of rp are asked for.
        constexpr int kStretch = (ROOMY ? 504 : 252) * G, kNeed = kStretch + 64, kFetchStep = 512;
        static_assert(kRing - kRingBlock - 2 * kFetchStep - kStretch >= kNeed, "a wait has to cover the next positions");
        int wait_at = 0, fetch_at = kFetchStep;
        auto keep_filled = [&]() {
            if (rp >= wait_at) {
                asm volatile("cp.async.wait_all;" ::: "memory");
                __syncwarp();
                wait_at = fetched >= 2 * nwords ? 0x7fffffff : (fetched - kNeed) / 2 + 1;
            }
            if (rp >= fetch_at) {
                __syncwarp();                                                  // readers of what is overwritten are done
                ring_fetch<kRing>(ring, src, 2 * nwords, rp, fetched, lane);
                fetch_at = rp + kFetchStep;
            }
        };
        for (int b = 0; b < n_batches; ++b) {
            meet();                                                   // the classes of batch b are there
            const int cnt = min(NP, P - b * NP);
            int* slot = slots + (b & 1) * NP * SW;
            SlotMeta* meta = sh.meta[b & 1];
            auto code = [&](const auto& find, int planes, int j) {
                int base[G], zz[G];
                if (pull_position<G>(planes, find, x, words, rp, lc, base, zz)) {
                    tail_put<G>(slot + j * SW + 32 * G, base);
                } else {
                    decode_position_escapes<G>(zz, planes, find, x, words, rp, lane);
                    if (lane == 0) meta[j].escaped = 1;
                }
                slot_put_ints<G>(slot + j * SW, lane, zz);
            };
            auto any_code = [&](const SlotMeta& m, int j) {
                if (m.table >= kWideFrom) code(WideLookup{tb.wide[m.table - kWideFrom]}, m.planes, j);
                else code(Lookup{tb.first[m.table], tb.fc[m.table]}, m.planes, j);
            };
            // One vote a batch: where all positions have wide tables, the loop has no other case, and two
            // positions share the check of the ring.
            if (ROOMY && !__any_sync(kFull, lane < cnt && (meta[lane].planes < 0 || meta[lane].table < kWideFrom))) {
#pragma unroll 1
                for (int j = 0; j < cnt; j += 2) {
                    const SlotMeta m0 = meta[j], m1 = meta[min(j + 1, cnt - 1)];
                    keep_filled();
                    code(WideLookup{tb.wide[m0.table - kWideFrom]}, m0.planes, j);
                    if (j + 1 < cnt) code(WideLookup{tb.wide[m1.table - kWideFrom]}, m1.planes, j + 1);
                }
            } else {
                SlotMeta next = meta[0];
#pragma unroll 1
                for (int j = 0; j < cnt; ++j) {
                    const SlotMeta m = next;
                    if (j + 1 < cnt) next = meta[j + 1];
                    if (m.planes < 0) continue;
                    keep_filled();
                    any_code(m, j);
                }
            }
        }
        meet();
        bad = bad || x != kRansL || rp != nwords;
        if (__any_sync(kFull, bad) && lane == 0) atomicOr(a.status, kStCorrupt);
        asm volatile("cp.async.wait_all;" ::: "memory");                       // of a damaged chunk: nothing may land later
    }
}

// GW: warps of a chunk's group, several groups a block (decoding where predictions come from memory: the coder's
// chain is all that takes time then, and one block of eight coders an SM shares the 33 KB of tables that keep blocks
// of one coder to four an SM), or 0: the block has one chunk.
constexpr int kGroupWarps = 4;
template <int D>
constexpr int kGroups = D == 256 ? 4 : 8;                // by the registers
// Warps of a block that has its SM to itself: 24 beside the coder (7 idle), since a prediction's latency (4000 cycles)
// is what an encoder waits for (2 x 512 positions of 64: 55 -> 43 us, 64 chunks of 256 x 128: 121 -> 92; with 12).
template <int D>
constexpr int kAloneWarps = D == 256 ? 16 : 32;
// 64 registers: the row loads of a prediction's whole unrolled batch are in flight before the first use.
// AHEAD: the call's variance terms were formed ahead; an instantiation of its own, since asking for each position costs
// registers (168 streams x 384 positions of 256, K = 128, uniform: 983 + 916 us with the question, 946 + 882 without; 1024 x
// 128 positions of 128: encoding 245 -> 240).
template <int D, bool DENSE, bool ENC, bool ROOMY, bool AHEAD = false, int GW = 0>
__global__ void __launch_bounds__(GW ? 32 * GW * kGroups<D> : ROOMY && !DENSE ? 32 * kAloneWarps<D> : 512, GW || D == 256 || (ROOMY && !DENSE) ? 1 : 2) coop_kernel(const CodecArgs a) {
    static_assert(GW == 0 || (DENSE && !ENC), "staging is addressed by block");
    using Tab = std::conditional_t<ENC, EncTables, WideDecTables>;
    __shared__ Tab tb;
    using Shared = CoopShared<GW ? GW - 1 : ROOMY ? coop_predictors(DENSE ? 16 : kAloneWarps<D>) : 7>;
    __shared__ Shared shared[GW ? kGroups<D> : 1];
    // Warps go to an SM's four schedulers in turn.  A block that has its SM to itself (16 warps or more) leaves the
    // coder's scheduler to the coder: the warps that would share it stay idle.  The coders of groups lie on
    // different schedulers.
    const int lane = threadIdx.x & 31, hw = threadIdx.x >> 5, warps = GW ? GW : (int)(blockDim.x >> 5), NP = coop_predictors(warps);   // NP predicting warps
    const int group = GW ? hw / GW : 0;
    const int warp = GW ? (hw - group) & (GW - 1) : NP < warps - 1 ? ((hw & 3) == 0 ? (hw == 0 ? 0 : -1) : hw - (hw >> 2)) : hw;
    const int Kp = DENSE ? 0 : a.sh.Kp;
    Shared& sh = shared[group];
    int2* pairs = GW ? reinterpret_cast<int2*>(reinterpret_cast<unsigned char*>(g_pair_smem) + group * coop_smem(GW, 0, D, DENSE, ENC, ROOMY)) : g_pair_smem;
    int* slots = reinterpret_cast<int*>(pairs + NP * 2 * Kp);                                // [2][NP] slots
    uint16_t* ring = reinterpret_cast<uint16_t*>(slots + 2 * NP * kDecSlotWords<Geo<D>::G>);  // decoding
    const Meet<GW> meet{group};
    const LaneCode lc = lane_code(lane);
    load_tables(&tb, ENC ? reinterpret_cast<const Tab*>(&a.tables->enc) : reinterpret_cast<const Tab*>(&a.tables->wide));
    chain_wait();
    const int Wl = DENSE ? a.dense_nt : 2 * a.sh.L * a.sh.H;
    const unsigned per_table = (unsigned)a.S * (unsigned)a.chunks, total = (unsigned)Wl * per_table;
    if (ENC) clear_unused_slots(a, DENSE ? a.dense_t0 : 0, Wl);
    QueueCursor qc = DENSE ? QueueCursor{0, 0} : queue_of_this_sm(a);
    auto all_meet = [&]() { if (GW) meet(); else __syncthreads(); };
    if (GW) __syncthreads();                                                   // the tables are there

    for (;;) {
        if (warp == 0) {
            const unsigned item = DENSE ? next_ticket(a.ticket, lane) : next_queued(a, qc, per_table, Wl, lane);
            if (lane == 0) {
                CoopItem ci{};
                ci.go = -1;
                if (item < total) {
                    ci.it = bulk_item(a, item, DENSE ? a.dense_t0 : 0);
                    ci.go = ci.it.P > 0;
                    ci.row0 = (long long)ci.it.s * a.n + ci.it.p0;
                    ci.kv0 = kv_elem(a.kv, ci.it.t, a.sh.H, ci.it.s, ci.it.p0);
                    if (ENC && !ci.go) { a.st.chunk_offset[ci.it.slot] = 0; a.st.chunk_bytes[ci.it.slot] = 0; }
                    if (!ENC && ci.go) {
                        ci.off = a.st.chunk_offset[ci.it.slot];
                        ci.nbytes = a.st.chunk_bytes[ci.it.slot];
                        if (ci.nbytes < 128u || (ci.nbytes & 1u) || (ci.off & 15ull) || ci.off + ci.nbytes > a.st.capacity) {
                            atomicOr(a.status, kStCorrupt);
                            ci.go = 0;
                        }
                    }
                }
                sh.item = ci;
            }
        }
        all_meet();
        const int go = sh.item.go;
        if (go < 0) break;
        if (go > 0) {
            if (warp == 0) coop_code<D, ENC, ROOMY, GW>(a, sh, tb, slots, ring, NP, meet, lc);
            else if (warp > 0) coop_predict<D, DENSE, ENC, AHEAD, GW>(a, sh, tb, pairs + (warp - 1) * 2 * Kp, slots, warp - 1, NP, meet, lc);
        }
        all_meet();                                                            // the chunk is coded; its item has been read
        if (ENC && go > 0 && sh.dst)
            copy_words(sh.dst, a.staging + (long long)blockIdx.x * a.staging_words_per_warp + sh.wp,
                       (int)a.staging_words_per_warp - sh.wp, threadIdx.x, blockDim.x);
    }
}

}  // namespace

// Four decoding blocks of eight warps fit an SM (228 KB, 1 KB of them each block's own) up to K = 100: with 512 bytes more a
// block three did, and 168 streams x 768 positions, K = 100, decoded in 652 us instead of 484.
static_assert(sizeof(WideDecTables) + sizeof(CoopShared<7>) + coop_smem(8, 100, 128, false, false, false) + 1024 <= 228 * 1024 / 4, "shared memory of a block");

cudaError_t launch_coop(const CodecArgs& a, bool encode, cudaStream_t st) {
    return dispatch_d(a.sh.d, [&](auto D) {
        constexpr int d = decltype(D)::value;
        const bool dense = a.mu_dense != nullptr;
        const long long items = (long long)(dense ? a.dense_nt : 2 * a.sh.L * a.sh.H) * a.S * a.chunks;
        // Seven warps beside the coder: with three the coder waits, with fifteen two coders an SM are too few
        // (encode + decode of 4096 positions x 128 streams: 2.9, 2.3 and 3.2 ms).  Where there is a chunk an SM at
        // most, a block of kAloneWarps, or of 16 (streamed predictions, and where the pairs of more do not fit).
        const int most = dense ? 16 : kAloneWarps<d>;
        const int fit = coop_smem(most, a.sh.Kp, d, dense, encode, true) <= kMostSmem ? most : 16;
        const bool alone = items <= sm_count() && coop_smem(fit, a.sh.Kp, d, dense, encode, true) <= kMostSmem;
        const bool roomy = dense || alone;
        // Coders alone with their chains: eight an SM, in groups of one block, once there are more chunks than the four
        // that blocks of eight warps hold (2048 chunks of 256 positions: 745 -> 548 us with 128 components, 1180 -> 703 with 256; 1024 of 128: 337 -> 252).
        if (dense && !encode && items > 4ll * sm_count()) {
            auto kern = coop_kernel<d, true, false, true, false, kGroupWarps>;
            const size_t smem = kGroups<d> * coop_smem(kGroupWarps, 0, d, true, false, true);
            const cudaError_t e = allow_smem(kern, smem);
            if (e != cudaSuccess) return e;
            count_launch();
            return launch_kernel(kern, (unsigned)sm_count(), 32 * kGroupWarps * kGroups<d>, smem, st, false, 1, a);
        }
        auto gather = [&](auto ahead) {
            constexpr bool A = decltype(ahead)::value;
            return roomy ? (encode ? coop_kernel<d, false, true, true, A> : coop_kernel<d, false, false, true, A>)
                         : (encode ? coop_kernel<d, false, true, false, A> : coop_kernel<d, false, false, false, A>);
        };
        auto kern = dense ? (encode ? coop_kernel<d, true, true, true> : coop_kernel<d, true, false, true>)
                  : a.s1 ? gather(std::true_type{}) : gather(std::false_type{});
        const int warps = alone ? fit : 8;
        const size_t smem = coop_smem(warps, a.sh.Kp, d, dense, encode, roomy);
        const cudaError_t e = allow_smem(kern, smem);
        if (e != cudaSuccess) return e;
        int occ = 1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, warps * 32, smem) != cudaSuccess || occ < 1) occ = 1;
        const long long blocks = std::min<long long>(items, (long long)sm_count() * occ);
        // chained where its blocks and the top-K's fit beside each other, a block an SM
        const bool chained = a.behind > 0 && a.behind + blocks <= sm_count();
        count_launch();
        return launch_kernel(kern, (unsigned)blocks, warps * 32, smem, st, chained, 1, a);
    });
}

}  // namespace plc
