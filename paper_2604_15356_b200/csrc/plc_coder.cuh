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
#pragma once
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
// Both, as a context keeps them in device memory.
struct CoderTables { EncTables enc; DecTables dec; };
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

// Words of the stream are written back to front: stage[wp - 1], stage[wp - 2], ...  In decoder order a
// step is: 2S plane words, the refill words of the lanes that renormalise (lanes ascending), the raw
// high parts of escaped lanes (lanes ascending, low half first).
template <int GP>
__device__ __forceinline__ void put_planes(const uint32_t* lo, const int* base, int S, uint16_t* __restrict__ stage, const LaneCode& lc) {
    uint32_t packed = 0;
#pragma unroll
    for (int i = 0; i < GP; ++i) packed |= lo[i] << (i * S);
    const uint32_t plane = transpose32(packed, lc);
    // lane j = i * S + b: plane b of step i, at halfword base[i] + 2 b = (base[i] - 2 i S) + 2 j
    int off[GP];
#pragma unroll
    for (int i = 0; i < GP; ++i) off[i] = base[i] - 2 * i * S;
    if (lc.lane < GP * S) {
        uint16_t* p = stage + (of_my_step<GP>(off, lc.lane, S) + 2 * lc.lane);
        p[0] = (uint16_t)plane;
        p[1] = (uint16_t)(plane >> 16);
    }
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

// All G components of one position, last component first; S bit planes a component (the same in all
// lanes).  Returns the new wp.
template <int G>
__device__ __forceinline__ int encode_position(const int (&sym)[G], int S, const EncEntry* tbl, uint32_t& x,
                                               uint16_t* __restrict__ stage, int wp, const LaneCode& lc, unsigned& n_escapes) {
    const int half = (1 << S) >> 1;                        // |sym| <= 2^30, S <= 15: no overflow
    int u[G];
    uint32_t at[G], worst = 0;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        u[g] = sym[g] + half;
        at[g] = (uint32_t)((u[g] >> S) + kHiMax);
        worst = max(worst, at[g]);
    }
    if (__any_sync(kFull, worst > 2u * kHiMax)) return encode_position_escapes<G>(u, S, tbl, x, stage, wp, lc.lane, n_escapes);
    EncEntry e[G];
#pragma unroll
    for (int g = 0; g < G; ++g) e[g] = tbl[at[g]];
    int base[G];
#pragma unroll
    for (int g = G - 1; g >= 0; --g) {
        const bool emit = x >= (e[g].fc << 17);            // f << 17: the count above f is shifted out
        const uint32_t emask = __ballot_sync(kFull, emit);
        wp -= __popc(emask);
        if (emit) stage[wp + __popc(emask & lc.lt)] = (uint16_t)x;
        x = push_state(x, emit, e[g]);
        wp -= 2 * S;
        base[g] = wp;
    }
    if (S > 0) {
        const uint32_t mask = (1u << S) - 1u;
        uint32_t lo[G];
#pragma unroll
        for (int g = 0; g < G; ++g) lo[g] = (uint32_t)u[g] & mask;
        if (G * S <= 32) put_planes<G>(lo, base, S, stage, lc);
        else if (G * S <= 64) {
            if constexpr (G >= 2) {
#pragma unroll
                for (int g = 0; g < G; g += G / 2) put_planes<G / 2>(lo + g, base + g, S, stage, lc);
            }
        } else {
            if constexpr (G >= 4) {
#pragma unroll
                for (int g = 0; g < G; g += G / 4) put_planes<G / 4>(lo + g, base + g, S, stage, lc);
            }
        }
    }
    return wp;
}

// Symbol of a slot: its fc entry and its place in the alphabet.
__device__ __forceinline__ uint32_t find_symbol(uint32_t x, const uint8_t* first, const uint32_t* fcs, int& zz) {
    const uint32_t slot = x & (kProbM - 1u);
    const float r = 8421376.0f - __uint_as_float(0x4b000000u | slot);      // 2^23 + 2^15 - (2^23 + slot), exact
    const int z = first[(__float_as_uint(r) >> 19) - 127u * 16u];
    const uint32_t a = fcs[z], b = fcs[z + 1];
    const bool next = slot >= (b >> 16);
    zz = next ? z + 1 : z;
    return next ? b : a;
}
__device__ __forceinline__ int hi_of(int zz) {                            // 0, +1, -1, +2, ...
    const int t = (zz + 1) >> 1;
    return (zz & 1) ? t : -t;
}

template <int GP, class Words>
__device__ __forceinline__ uint32_t get_planes(const int* base, int S, const Words& words, const LaneCode& lc) {
    int off[GP];
#pragma unroll
    for (int i = 0; i < GP; ++i) off[i] = base[i] - 2 * i * S;
    uint32_t plane = 0;
    if (lc.lane < GP * S) {
        const int p = of_my_step<GP>(off, lc.lane, S) + 2 * lc.lane;
        plane = words(p) | (words(p + 1) << 16);
    }
    return transpose32(plane, lc);
}

// Positions with an escaped component, one step at a time.
template <int G, class Words>
__device__ __forceinline__ void decode_position_escapes(int (&sym)[G], int S, const uint8_t* first, const uint32_t* fcs, uint32_t& x,
                                                        const Words& words, int& rp, int lane) {
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
        const uint32_t fc = find_symbol(x, first, fcs, zz);
        x = (fc & 0xffffu) * (x >> kProbBits) + (x & (kProbM - 1u)) - (fc >> 16);
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

// All G components of one position.  words(i) reads 16-bit word i of the chunk (any i: the reader keeps
// the access in bounds; rp advances regardless, so the caller's final check of rp reports a short chunk).
template <int G, class Words>
__device__ __forceinline__ void decode_position(int (&sym)[G], int S, const uint8_t* first, const uint32_t* fcs, uint32_t& x,
                                                const Words& words, int& rp, const LaneCode& lc) {
    const uint32_t x0 = x;
    const int rp0 = rp;
    int base[G], hi[G];
    bool esc = false;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        base[g] = rp;
        rp += 2 * S;
        int zz;
        const uint32_t fc = find_symbol(x, first, fcs, zz);
        x = (fc & 0xffffu) * (x >> kProbBits) + (x & (kProbM - 1u)) - (fc >> 16);
        const bool need = x < kRansL;
        const uint32_t nmask = __ballot_sync(kFull, need);
        if (need) x = (x << 16) | words(rp + __popc(nmask & lc.lt));
        rp += __popc(nmask);
        esc = esc || zz == kEsc;
        hi[g] = hi_of(zz);
    }
    if (__any_sync(kFull, esc)) {                          // the words after the first escape were read wrongly: start over
        x = x0; rp = rp0;
        decode_position_escapes<G, Words>(sym, S, first, fcs, x, words, rp, lc.lane);
        return;
    }
    if (S == 0) {
#pragma unroll
        for (int g = 0; g < G; ++g) sym[g] = hi[g];
        return;
    }
    const uint32_t mask = (1u << S) - 1u, half = (1u << S) >> 1;
    auto join = [&](int g, uint32_t lo) { sym[g] = (int)(((uint32_t)hi[g] << S) + (lo & mask) - half); };
    if (G * S <= 32) {
        const uint32_t v = get_planes<G>(base, S, words, lc);
#pragma unroll
        for (int g = 0; g < G; ++g) join(g, v >> (g * S));
    } else if (G * S <= 64) {
        if constexpr (G >= 2) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t v = get_planes<G / 2>(base + h * (G / 2), S, words, lc);
#pragma unroll
                for (int g = 0; g < G / 2; ++g) join(h * (G / 2) + g, v >> (g * S));
            }
        }
    } else {
        if constexpr (G >= 4) {
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const uint32_t v = get_planes<G / 4>(base + h * (G / 4), S, words, lc);
#pragma unroll
                for (int g = 0; g < G / 4; ++g) join(h * (G / 4) + g, v >> (g * S));
            }
        }
    }
}

#endif  // __CUDACC__
}  // namespace plc
