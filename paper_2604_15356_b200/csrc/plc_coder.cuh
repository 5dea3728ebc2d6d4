// The interleaved rANS coder of one position (32 lanes, G components a lane, one shared word stream),
// shared by the kernels of plc_codec.cu and plc_coop.cu.
//
// What bounds a coder warp is its serial chain (the state x, then the word cursor) and, in full
// grids, issue slots.  Three things keep both short:
//   * the G steps of a position are straight-line code: escapes (a component beyond the alphabet) are
//     looked for once per position and take a step-by-step route of their own, so the table look-ups
//     of all steps are issued together and nothing of a step waits for a vote of the step before;
//   * the raw bit planes of all G steps are moved by ONE 32 x 32 bit transpose across the warp (five
//     shuffles): lane j then holds plane j mod S of step j / S whole, so a position costs two stores
//     (or loads) instead of one ballot, test and store per plane;
//   * the decoder finds a slot's symbol in two dependent look-ups instead of a six-step binary search:
//     r = 2^15 - slot as a binary32 number, its exponent and top four mantissa bits index a byte table
//     that holds the smallest symbol of that interval, and no interval of any of the 40 tables holds
//     more than one symbol boundary (checked on the host for every slot when the tables are built).
//     The eight tables that positions with bit planes use also exist in a wide form with everything an
//     interval needs in one 8-byte entry (kernels with one coder a block have room for it).
// Cycles of one warp alone, four steps with four planes each: encoding 618 before the state's chain was
// taken out of the words' places, decoding 1080 before the wide form and the refill window.
#pragma once
#include <type_traits>

#include "plc_common.cuh"

namespace plc {

// Encoder tables are indexed by hi + 31 (hi in [-31, 31]; entry 63 = escape): the symbol's place in
// the alphabet (0, +1, -1, +2, ...) only matters for the cumulative counts, which are kept.
struct EncTables { EncEntry enc[kNumTables][kNumSym]; };
// Decoder tables: first[] = smallest symbol of an interval of r (see above), fc[] = f | (c << 16), one
// entry past the escape with c = 2^15.
constexpr int kFcStride = kNumSym + 4;
struct DecTables { uint8_t first[kNumTables][256]; uint32_t fc[kNumTables][kFcStride]; };
static_assert(sizeof(EncTables) % 16 == 0 && sizeof(DecTables) % 16 == 0, "tables are copied in 16-byte pieces");
// Decoder tables with the wide form (f0 | c0 << 16, f1 | z0 << 16: an interval's first symbol z0 and the
// next) for table ids 8 .. 15, the ids of classes with bit planes; the others as above.
constexpr int kWideFrom = 8 - kQMin;
struct WideDecTables { uint8_t first[kWideFrom][256]; uint32_t fc[kWideFrom][kFcStride]; uint2 wide[kNumTables - kWideFrom][256]; };
static_assert(sizeof(WideDecTables) % 16 == 0, "tables are copied in 16-byte pieces");
// All of them, as a context keeps them in device memory.
struct CoderTables { EncTables enc; DecTables dec; WideDecTables wide; };
bool build_coder_tables(CoderTables* t);             // host; false if an interval held two boundaries

#ifdef __CUDACC__

// Block-wide copy of a table set into shared memory (followed by __syncthreads in the caller).
template <class Tab>
__device__ __forceinline__ void load_tables(Tab* dst, const Tab* __restrict__ src) {
    const uint4* s = reinterpret_cast<const uint4*>(src);
    uint4* d = reinterpret_cast<uint4*>(dst);
    for (int i = threadIdx.x; i < (int)(sizeof(Tab) / 16); i += blockDim.x) d[i] = __ldg(s + i);
}

// Per-lane constants of the coder.
struct LaneCode {
    int lane;
    uint32_t lt;             // lanes below this one
    uint32_t sel16, sel8;    // byte selectors of the transpose's first two stages
};
__device__ __forceinline__ LaneCode lane_code(int lane) {
    LaneCode lc;
    lc.lane = lane; lc.lt = lanemask_lt();
    lc.sel16 = (lane & 16) ? 0x3276u : 0x5410u;
    lc.sel8 = (lane & 8) ? 0x3715u : 0x6240u;
    return lc;
}

// 32 x 32 bit transpose across the warp: bit j of lane l's word becomes bit l of lane j's.
template <int O>
__device__ __forceinline__ uint32_t transpose_stage(uint32_t x, int lane) {
    constexpr uint32_t B = O == 4 ? 0x0f0f0f0fu : O == 2 ? 0x33333333u : 0x55555555u;   // bits whose index has bit O clear
    const uint32_t y = __shfl_xor_sync(kFull, x, O);
    const bool up = (lane & O) != 0;
    const uint32_t keep = up ? ~B : B;
    const uint32_t rot = __funnelshift_l(y, y, up ? 32 - O : O);
    return (x & keep) | (rot & ~keep);
}
__device__ __forceinline__ uint32_t transpose32(uint32_t x, const LaneCode& lc) {
    x = __byte_perm(x, __shfl_xor_sync(kFull, x, 16), lc.sel16);
    x = __byte_perm(x, __shfl_xor_sync(kFull, x, 8), lc.sel8);
    x = transpose_stage<4>(x, lc.lane);
    x = transpose_stage<2>(x, lc.lane);
    return transpose_stage<1>(x, lc.lane);
}

// at[i] of the lane's own step lane / S among the GP steps of a group, by comparisons (S is uniform).
template <int GP>
__device__ __forceinline__ int of_my_step(const int* at, int lane, int S) {
    int v = at[0];
#pragma unroll
    for (int i = 1; i < GP; ++i) v = lane >= i * S ? at[i] : v;
    return v;
}

// State update of one encoder step: emits the low half of x if it would overflow, then codes e.
__device__ __forceinline__ uint32_t push_state(uint32_t x, bool emit, EncEntry e) {
    const uint32_t f = e.fc & 0xffffu, mf = kProbM - f;
    const uint32_t xe = emit ? x >> 16 : x;
    const uint32_t q = __umulhi(xe, e.rcp);               // floor(xe / f) or one less
    const uint32_t r = xe - q * f;
    const uint32_t y = xe + (e.fc >> 16) + q * mf;        // (q << 15) + r + c
    return r >= f ? y + mf : y;
}

// The planes of a position travel in groups of GP steps whose planes fit one transpose (GP * S <= 32);
// plane_group<G>(S) is that GP, kPlaneWords<G> the most groups a position has (S <= 15).
template <int G>
constexpr int kPlaneWords = G <= 2 ? 1 : G / 2;
template <int G, class F>
__device__ __forceinline__ void by_plane_group(int S, F&& f) {             // calls f(integral_constant<GP>)
    if (G <= 2 || G * S <= 32) f(std::integral_constant<int, G>{});
    else if (G == 4 || G * S <= 64) f(std::integral_constant<int, (G >= 2 ? G / 2 : 1)>{});
    else f(std::integral_constant<int, (G >= 4 ? G / 4 : 1)>{});
}

// What a position's symbols put into the stream, before the state is known: table entries and, per
// group, lane j's plane.
template <int G>
struct Prepared {
    EncEntry e[G];
    uint32_t plane[kPlaneWords<G>];
};
template <int G>
__device__ __forceinline__ void prepare_position(const int (&u)[G], const uint32_t (&at)[G], int S, const EncEntry* tbl, const LaneCode& lc,
                                                 Prepared<G>& pr) {
#pragma unroll
    for (int g = 0; g < G; ++g) pr.e[g] = tbl[at[g]];
#pragma unroll
    for (int i = 0; i < kPlaneWords<G>; ++i) pr.plane[i] = 0;
    if (S > 0) {
        const uint32_t mask = (1u << S) - 1u;
        by_plane_group<G>(S, [&](auto gp) {
            constexpr int GP = decltype(gp)::value;
#pragma unroll
            for (int i = 0; i < G / GP; ++i) {
                uint32_t packed = 0;
#pragma unroll
                for (int k = 0; k < GP; ++k) packed |= ((uint32_t)u[i * GP + k] & mask) << (k * S);
                pr.plane[i] = transpose32(packed, lc);
            }
        });
    }
}

// Splits symbols (S planes a component) into u = sym + 2^(S-1) and table places; true if none escapes.
template <int G>
__device__ __forceinline__ bool split_symbols(const int (&sym)[G], int S, int (&u)[G], uint32_t (&at)[G]) {
    const int half = (1 << S) >> 1;                        // |sym| <= 2^30, S <= 15: no overflow
    uint32_t worst = 0;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        u[g] = sym[g] + half;
        at[g] = (uint32_t)((u[g] >> S) + kHiMax);
        worst = max(worst, at[g]);
    }
    return !__any_sync(kFull, worst > 2u * kHiMax);
}

// The serial part of coding a position: the state through its steps, last component first.  low[g], emask[g]:
// the state before step g and the lanes whose low half goes into the stream there.
template <int G>
__device__ __forceinline__ void chain_position(const EncEntry (&e)[G], uint32_t& x, uint32_t (&low)[G], uint32_t (&emask)[G], bool (&emit)[G]) {
#pragma unroll
    for (int g = G - 1; g >= 0; --g) {
        emit[g] = x >= (e[g].fc << 17);                    // f << 17: the count above f is shifted out
        emask[g] = __ballot_sync(kFull, emit[g]);
        low[g] = x;
        x = push_state(x, emit[g], e[g]);
    }
}
// Words a position takes.
template <int G>
__device__ __forceinline__ int words_of(const uint32_t (&emask)[G], int S) {
    int n = 2 * S * G;
#pragma unroll
    for (int g = 0; g < G; ++g) n += __popc(emask[g]);
    return n;
}
// The rest: its words to stage[base ...].  In decoder order a step is: 2S plane words, the refill words of the
// lanes that renormalise (lanes ascending), the raw high parts of escaped lanes (lanes ascending, low
// half first).
template <int G>
__device__ __forceinline__ void place_position(const uint32_t (&plane)[kPlaneWords<G>], const uint32_t (&low)[G], const uint32_t (&emask)[G],
                                               const bool (&emit)[G], int S, uint16_t* __restrict__ stage, int base, const LaneCode& lc) {
    int first[G];                                          // lane j = g S + b of a group: halfword first + 2 j
#pragma unroll
    for (int g = 0; g < G; ++g) {
        first[g] = base - 2 * S * g;
        base += 2 * S;
        if (emit[g]) stage[base + __popc(emask[g] & lc.lt)] = (uint16_t)low[g];
        base += __popc(emask[g]);
    }
    if (S > 0)
        by_plane_group<G>(S, [&](auto gp) {
            constexpr int GP = decltype(gp)::value;
#pragma unroll
            for (int i = 0; i < G / GP; ++i) {
                if (lc.lane < GP * S) {
                    uint16_t* p = stage + (of_my_step<GP>(first + i * GP, lc.lane, S) + 2 * (i * GP * S + lc.lane));
                    p[0] = (uint16_t)plane[i];
                    p[1] = (uint16_t)(plane[i] >> 16);
                }
            }
        });
}

// Positions with an escaped component, one step at a time.
template <int G>
__device__ __forceinline__ int encode_position_escapes(const int (&u)[G], int S, const EncEntry* tbl, uint32_t& x,
                                                       uint16_t* __restrict__ stage, int wp, int lane, unsigned& n_escapes) {
    const uint32_t lt = lanemask_lt();
#pragma unroll 1
    for (int g = G - 1; g >= 0; --g) {
        int ug = u[0];
#pragma unroll
        for (int i = 1; i < G; ++i) ug = g == i ? u[i] : ug;
        const int hi = ug >> S;
        const uint32_t at = (uint32_t)(hi + kHiMax);
        const bool esc = at > 2u * kHiMax;
        const EncEntry e = tbl[min(at, (uint32_t)kEsc)];
        const bool emit = x >= (e.fc << 17);
        const uint32_t emask = __ballot_sync(kFull, emit), xmask = __ballot_sync(kFull, esc);
        wp -= 2 * S + __popc(emask) + 2 * __popc(xmask);
        if (esc) {
            const int w = wp + 2 * S + __popc(emask) + 2 * __popc(xmask & lt);
            stage[w] = (uint16_t)((uint32_t)hi & 0xffffu);
            stage[w + 1] = (uint16_t)((uint32_t)hi >> 16);
        }
        n_escapes += __popc(xmask);
        if (emit) stage[wp + 2 * S + __popc(emask & lt)] = (uint16_t)x;
        x = push_state(x, emit, e);
#pragma unroll 1
        for (int b = 0; b < S; ++b) {
            const uint32_t plane = __ballot_sync(kFull, (ug >> b) & 1);
            if (lane < 2) stage[wp + 2 * b + lane] = (uint16_t)(plane >> (16 * lane));
        }
    }
    return wp;
}

// All G components of one position; S bit planes a component (the same in all lanes).
template <int G>
__device__ __forceinline__ int encode_position(const int (&sym)[G], int S, const EncEntry* tbl, uint32_t& x,
                                               uint16_t* __restrict__ stage, int wp, const LaneCode& lc, unsigned& n_escapes) {
    int u[G];
    uint32_t at[G];
    if (!split_symbols<G>(sym, S, u, at)) return encode_position_escapes<G>(u, S, tbl, x, stage, wp, lc.lane, n_escapes);
    Prepared<G> pr;
    prepare_position<G>(u, at, S, tbl, lc, pr);
    uint32_t low[G], emask[G];
    bool emit[G];
    chain_position<G>(pr.e, x, low, emask, emit);
    wp -= words_of<G>(emask, S);
    place_position<G>(pr.plane, low, emask, emit, S, stage, wp, lc);
    return wp;
}

// One decoder step before its refill: the symbol (place in the alphabet) of state x and the next state.
// r = 2^15 - slot as a float: 2^23 + 2^15 - (2^23 + slot), exact; its bits from the fourth mantissa bit up
// number the intervals.
__device__ __forceinline__ int interval_of(uint32_t slot) {
    const float r = 8421376.0f - __uint_as_float(0x4b000000u | slot);
    return (int)(__float_as_uint(r) >> 19) - 127 * 16;
}
struct Lookup {                                            // any table: two dependent look-ups
    const uint8_t* first;
    const uint32_t* fc;
    __device__ __forceinline__ uint32_t operator()(uint32_t x, int& zz) const {
        const uint32_t slot = x & (kProbM - 1u);
        const int z = first[interval_of(slot)];
        const uint32_t a = fc[z], b = fc[z + 1];
        const bool next = slot >= (b >> 16);
        zz = next ? z + 1 : z;
        const uint32_t e = next ? b : a;
        return (e & 0xffffu) * (x >> kProbBits) + slot - (e >> 16);
    }
};
struct WideLookup {                                        // tables kept in wide form: one
    const uint2* t;
    __device__ __forceinline__ uint32_t operator()(uint32_t x, int& zz) const {
        const uint32_t slot = x & (kProbM - 1u);
        const uint2 w = t[interval_of(slot)];
        const uint32_t f0 = w.x & 0xffffu, d = slot - (w.x >> 16), top = x >> kProbBits;
        const bool next = d >= f0;
        zz = (int)(w.y >> 16) + next;
        return next ? (w.y & 0xffffu) * top + (d - f0) : f0 * top + d;
    }
};
__device__ __forceinline__ int hi_of(int zz) {                            // 0, +1, -1, +2, ...
    const int t = (zz + 1) >> 1;
    return (zz & 1) ? t : -t;
}

// Positions with an escaped component, one step at a time.
template <int G, class Find, class Words>
__device__ __forceinline__ void decode_position_escapes(int (&sym)[G], int S, const Find& find, uint32_t& x, const Words& words, int& rp, int lane) {
    const uint32_t lt = lanemask_lt();
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
        uint32_t lo = 0;
#pragma unroll 1
        for (int b = 0; b < S; ++b) {
            const uint32_t w = words(rp + 2 * b + (lane >> 4));
            lo |= ((w >> (lane & 15)) & 1u) << b;
        }
        rp += 2 * S;
        int zz;
        x = find(x, zz);
        const bool need = x < kRansL;
        const uint32_t nmask = __ballot_sync(kFull, need);
        if (need) x = (x << 16) | words(rp + __popc(nmask & lt));
        rp += __popc(nmask);
        int hi = hi_of(zz);
        const bool esc = zz == kEsc;
        const uint32_t xmask = __ballot_sync(kFull, esc);
        if (esc) {
            const int at = rp + 2 * __popc(xmask & lt);
            hi = (int)(words(at) | (words(at + 1) << 16));
        }
        rp += 2 * __popc(xmask);
        const int v = (int)(((uint32_t)hi << S) + lo - ((1u << S) >> 1));
#pragma unroll
        for (int i = 0; i < G; ++i) sym[i] = g == i ? v : sym[i];
    }
}

// The serial part of decoding a position: advances x and rp, gives every step's place in the word
// stream and symbol (place in the alphabet); false if a component escaped (x and rp are then as before the call).
// words(i) reads 16-bit word i of the chunk (any i: the reader keeps the access in bounds; rp advances
// regardless, so the caller's final check of rp reports a short chunk).
template <int G, class Find, class Words>
__device__ __forceinline__ bool pull_position(int S, const Find& find, uint32_t& x, const Words& words, int& rp, const LaneCode& lc,
                                              int (&base)[G], int (&zz)[G]) {
    const uint32_t x0 = x;
    const int rp0 = rp;
    int top = 0;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        base[g] = rp;
        rp += 2 * S;
        const uint32_t window = words(rp + lc.lane);       // the step's refill words, fetched beside the look-up
        x = find(x, zz[g]);
        const bool need = x < kRansL;
        const uint32_t nmask = __ballot_sync(kFull, need);
        const uint32_t word = __shfl_sync(kFull, window, __popc(nmask & lc.lt));
        x = need ? (x << 16) | word : x;
        rp += __popc(nmask);
        top = max(top, zz[g]);
    }
    if (!__any_sync(kFull, top == kEsc)) return true;
    x = x0; rp = rp0;                                      // the words after the first escape were read wrongly
    return false;
}

// The rest: a position's planes from the word stream, and its symbols.
template <int G, class Words>
__device__ __forceinline__ void join_position(const int (&base)[G], const int (&zz)[G], int S, const Words& words, const LaneCode& lc, int (&sym)[G]) {
    if (S == 0) {
#pragma unroll
        for (int g = 0; g < G; ++g) sym[g] = hi_of(zz[g]);
        return;
    }
    const uint32_t mask = (1u << S) - 1u, half = (1u << S) >> 1;
    by_plane_group<G>(S, [&](auto gp) {
        constexpr int GP = decltype(gp)::value;
#pragma unroll
        for (int i = 0; i < G / GP; ++i) {
            int off[GP];
#pragma unroll
            for (int k = 0; k < GP; ++k) off[k] = base[i * GP + k] - 2 * k * S;
            uint32_t plane = 0;
            if (lc.lane < GP * S) {
                const int p = of_my_step<GP>(off, lc.lane, S) + 2 * lc.lane;
                plane = words(p) | (words(p + 1) << 16);
            }
            const uint32_t v = transpose32(plane, lc);
#pragma unroll
            for (int k = 0; k < GP; ++k) sym[i * GP + k] = (int)(((uint32_t)hi_of(zz[i * GP + k]) << S) + ((v >> (k * S)) & mask) - half);
        }
    });
}

// All G components of one position.
template <int G, class Find, class Words>
__device__ __forceinline__ void decode_position(int (&sym)[G], int S, const Find& find, uint32_t& x, const Words& words, int& rp,
                                                const LaneCode& lc) {
    int base[G], zz[G];
    if (pull_position<G>(S, find, x, words, rp, lc, base, zz)) join_position<G>(base, zz, S, words, lc, sym);
    else decode_position_escapes<G>(sym, S, find, x, words, rp, lc.lane);
}

#endif  // __CUDACC__
}  // namespace plc
