// Device functions shared by the kernels that predict and code: the gather of a position's mixture, the
// quantiser, work items and queues, vector loads and stores, the finishing of a chunk.
#pragma once
#include <type_traits>

#include "plc_coder.cuh"

namespace plc {
namespace {

template <int D>
struct Geo {
    static constexpr int R = D / 8;        // lanes that cover one row with 16-byte loads
    static constexpr int G = D / 32;       // components a lane owns
    static constexpr int ROWS = 32 / R;    // rows fetched by one warp-wide load
};

// component owned by (lane, g): 8 (lane mod R) + G (lane div R) + g
template <int D>
__device__ __forceinline__ int first_comp(int lane) {
    return 8 * (lane % Geo<D>::R) + Geo<D>::G * (lane / Geo<D>::R);
}

// Sum of squares of the lane's G values, then over the warp; the same chain is used for the row
// norms and for ||mu||^2 so that a point-mass mixture has exactly zero variance.
template <int G>
__device__ __forceinline__ float warp_norm2(const float (&v)[G]) {
    float p = 0.f;
#pragma unroll
    for (int g = 0; g < G; ++g) p = __fmaf_rn(v[g], v[g], p);
    return warp_sum(p);
}

// The values that a lane has loaded (two words of two), as binary32, through the tensor cores: in a product
// with the 8 x 8 identity, a lane's share of the 16 x 8 operand and its share of the result are the same
// elements, so the lanes need not hold anything that belongs together.  Every sum has one term that is not zero:
// exact for finite values (zeros come out as +0), infinities and NaN would reach other lanes.
__device__ __forceinline__ uint32_t widen_operand(int lane) {
    const int row = 2 * (lane & 3), col = lane >> 2;         // elements (row, col), (row + 1, col) of the identity
    return (row == col ? 0x3c00u : 0u) | (row + 1 == col ? 0x3c000000u : 0u);
}
__device__ __forceinline__ void widen(uint32_t lo, uint32_t hi, uint32_t operand, unsigned long long& a, unsigned long long& b) {
    float f0, f1, f2, f3;
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%7,%7,%7,%7};"
        : "=f"(f0), "=f"(f1), "=f"(f2), "=f"(f3) : "r"(lo), "r"(hi), "r"(operand), "f"(0.f));
    a = pack2(f0, f1); b = pack2(f2, f3);
}
// acc2 += w * (8 components of a row): four pairs.
template <bool WIDEN>
__device__ __forceinline__ void add_row(const char* p, float w, uint32_t operand, unsigned long long (&acc2)[4]) {
    const uint4 r = __ldg(reinterpret_cast<const uint4*>(p));
    const unsigned long long ww = pack2(w, w);
    if constexpr (WIDEN) {
        unsigned long long v[4];
        widen(r.x, r.y, operand, v[0], v[1]);
        widen(r.z, r.w, operand, v[2], v[3]);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc2[j] = fma2(ww, v[j], acc2[j]);
    } else {
        const __half2* hp = reinterpret_cast<const __half2*>(&r);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = __half22float2(hp[j]);
            acc2[j] = fma2(ww, pack2(f.x, f.y), acc2[j]);
        }
    }
}
// Mixture of one position for one table.  sp: the position's Kp pairs in shared memory (put_pair: byte
// offset of the candidate's row and weight, the Kp / ROWS entries of each row group together), Kp a
// multiple of 2 ROWS (the padding has weight 0 and a valid offset).  table, n2: the table's rows and
// their squared norms, s1_at: the position's variance term where it was formed ahead
// (launch_variance), or null; the same pointers in every lane.
// What bounds it: issue slots (per row and lane 8 conversions, 4 packed FMAs, a load), with the rows'
// latency on top; pairs are read two at a time and hold byte offsets, so that a row costs one addition
// beside its load.
// WIDEN: the conversions on the tensor cores, 2 instructions for 8 on the pipe that the packed FMAs need too (392
// of the 570 instructions that 64 rows of 128 take); for finite T and pairs that hold byte offsets.  Where it pays:
// see launch_rotq.  The coder's kernels lose more to the tensor instructions' latency than they gain (32 heads of
// 128, 8 layers, 16384 positions: 20.6 -> 21.8 ms at 64 registers, 25.2 at 48 with more warps).
// LANE_BASE: a row's address as the lane's own 64-bit base and the offset, one addition of three fewer, but two
// registers more.  It pays beside WIDEN and in the block-per-chunk kernel (128 streams x 4096 positions, both calls 1977 ->
// 1933 us, 3 x 333 x 64 streams 282 -> 275, although encoding then spills 46 bytes for 26), with 256 components only where the
// variance terms were formed ahead; the others lose loads in flight (131072 positions x 64 streams: decode 13.5 -> 15.5 ms).
// SHORT: straight-line stretches of 16 rows at most.
template <int D, bool WIDEN = false, bool LANE_BASE = WIDEN, bool SHORT = WIDEN>
__device__ __forceinline__ void predict(const char* __restrict__ table, const float* __restrict__ n2, const float* s1_at, bool pair_index,
                                        const int2* sp, int Kp, int lane, float inv_d,
                                        float (&mu)[Geo<D>::G], float& sigma2) {
    constexpr int R = Geo<D>::R, G = Geo<D>::G, ROWS = Geo<D>::ROWS;
    const int h = lane / R, iters = Kp / ROWS;
    const uint32_t lane_off = 16u * (lane % R);
    const char* lane_table = LANE_BASE ? table + lane_off : table;
    auto row_at = [&](int off) { return LANE_BASE ? lane_table + (uint32_t)off : table + ((uint32_t)off + lane_off); };
    // variance term first: its row-norm loads are in flight while the rows are gathered
    float s1 = 0.f;
    if (s1_at) {                                  // formed ahead: lane 0 brings the sum into the butterfly below
        if (lane == 0) s1 = __ldg(s1_at);
    } else {
        for (int k = lane; k < Kp; k += 32) {
            const int2 pr = sp[(k % ROWS) * iters + k / ROWS];
            const uint32_t at = pair_index ? (uint32_t)pr.x : (uint32_t)pr.x / (2u * D);
            s1 = __fmaf_rn(__int_as_float(pr.y), __ldg(n2 + at), s1);
        }
    }
    unsigned long long acc2[4] = {0ull, 0ull, 0ull, 0ull};   // four pairs of +0.f
    if (WIDEN || !pair_index) {
        const uint32_t operand = WIDEN ? widen_operand(lane) : 0u;
        // Straight-line stretches of 32, 16 and 8 rows: the loads of a stretch are issued as far ahead as the
        // kernel's registers allow (64 rows of 128 components, uniform candidates, 24 warps an SM: 8.0 ms
        // with stretches of 8 only, 6.4 ms with 32).
        const int4* pl = reinterpret_cast<const int4*>(sp + h * iters);
        int left = iters >> 1;
        auto rows = [&](auto count) {
            constexpr int N = decltype(count)::value;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int4 pr = pl[i];
                add_row<WIDEN>(row_at(pr.x), __int_as_float(pr.y), operand, acc2);
                add_row<WIDEN>(row_at(pr.z), __int_as_float(pr.w), operand, acc2);
            }
            pl += N;
            left -= N;
        };
        if constexpr (SHORT) {
#pragma unroll 1
            while (left >= 8) rows(std::integral_constant<int, 8>{});
        } else {
#pragma unroll 1
            while (left >= 16) rows(std::integral_constant<int, 16>{});
            if (left >= 8) rows(std::integral_constant<int, 8>{});
        }
        if (left >= 4) rows(std::integral_constant<int, 4>{});
#pragma unroll 1
        while (left > 0) rows(std::integral_constant<int, 1>{});
    } else {                                                 // tables of 4 GB or more: 64-bit offsets
#pragma unroll 1
        for (int it = 0; it < iters; ++it) {
            const int2 pr = sp[h * iters + it];
            add_row<false>(table + ((size_t)(uint32_t)pr.x * (2 * D) + lane_off), __int_as_float(pr.y), 0u, acc2);
        }
    }
    float acc[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) unpack2(acc2[j], acc[2 * j], acc[2 * j + 1]);
    // reduce-scatter over the ROWS lanes that hold partial sums of the same 8 components
    int cnt = 8;
#pragma unroll
    for (int o = (ROWS / 2) * R; o >= R; o >>= 1) {
        const bool up = (h & (o / R)) != 0;
        const int half = cnt / 2;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i < half) {
                float send = up ? acc[i] : acc[i + half];
                float keep = up ? acc[i + half] : acc[i];
                acc[i] = keep + __shfl_xor_sync(kFull, send, o);
            }
        }
        cnt = half;
    }
    float s2 = 0.f;
#pragma unroll
    for (int g = 0; g < G; ++g) { mu[g] = acc[g]; s2 = __fmaf_rn(mu[g], mu[g], s2); }
    // variance: (sum_k w_k ||T_k||^2 - ||mu||^2) / d.  Both sums over the warp in one butterfly: after the
    // first exchange the lower half-warp carries s1 and the upper s2 (the additions are warp_sum's, so a
    // point-mass mixture has exactly zero variance).
    const bool up = (lane & 16) != 0;
    float v = (up ? s2 : s1) + __shfl_xor_sync(kFull, up ? s1 : s2, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    const float other = __shfl_xor_sync(kFull, v, 16);
    sigma2 = fmaxf(0.f, (up ? other - v : v - other) * inv_d);
}

// The pairs of a position are brought into the warp's shared-memory slot with cp.async, one
// position ahead of their use and without passing through registers (two slots per warp): two entries
// (16 bytes) per copy, Kp is even.
__device__ __forceinline__ void prefetch_pairs(int2* sp, const int2* __restrict__ gp, int Kp, int lane) {
    for (int k = 2 * lane; k < Kp; k += 64) {
        const unsigned dst = (unsigned)__cvta_generic_to_shared(sp + k);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(gp + k) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
// Waits for this lane's copies (all but the newest `pending` groups), then makes the whole warp's
// copies visible to every lane.
template <int PENDING>
__device__ __forceinline__ void pairs_ready() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
    __syncwarp();
}

__device__ __forceinline__ int scale_class(float sigma2, float floor2, float inv_delta2) {
    return class_from_v((sigma2 + floor2) * inv_delta2);
}

// Lane 0's value for the whole warp, through a warp reduction: the result is provably the same in
// every lane, so everything derived from it (loop bounds, table addresses, branches) is kept out of
// the per-lane registers and needs no divergence handling.
__device__ __forceinline__ unsigned from_lane0(unsigned v, int lane) {
    return __reduce_or_sync(kFull, lane == 0 ? v : 0u);
}
__device__ __forceinline__ unsigned next_ticket(unsigned int* ticket, int lane) {
    unsigned t = 0;
    if (lane == 0) t = atomicAdd(ticket, 1u);
    return from_lane0(t, lane);
}

// Work queues of the gather kernels.  The tables are dealt round-robin to nq queues (queue k owns
// tables k, k + nq, ...), each queue lists its (table, session, chunk) items table-major, and the
// g SMs with the same smid / g serve one queue.  The warps resident on an SM therefore gather from
// one or two tables at a time, so candidate rows that several positions share are found in that
// SM's L1, and the number of tables in flight on the whole GPU stays near nq.  A warp whose queue
// is empty moves on to the next queue (and never returns), so the tail is balanced by stealing.
// Returns the item in table-major numbering (table * per_table + rest), or ~0u when all is taken.
__device__ __forceinline__ unsigned smid() {
    unsigned r;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
    return r;
}
struct QueueCursor { int q, tried; };
__device__ __forceinline__ QueueCursor queue_of_this_sm(const CodecArgs& a) {
    QueueCursor qc;
    qc.q = (int)((smid() / (unsigned)a.sched_g) % (unsigned)a.sched_nq);   // fewer tables than SM groups: spread the groups evenly
    qc.tried = 0;
    return qc;
}
__device__ __forceinline__ unsigned next_queued(const CodecArgs& a, QueueCursor& qc, unsigned per_table, int n_tables, int lane) {
    unsigned item = ~0u;
    if (lane == 0) {
        while (qc.tried < a.sched_nq) {
            const unsigned nt = (unsigned)max(0, (n_tables - qc.q + a.sched_nq - 1) / a.sched_nq);
            const unsigned j = atomicAdd(a.ticket + qc.q, 1u);
            if (j < nt * per_table) {
                item = ((unsigned)qc.q + (unsigned)a.sched_nq * (j / per_table)) * per_table + j % per_table;
                break;
            }
            qc.q = qc.q + 1 == a.sched_nq ? 0 : qc.q + 1;
            ++qc.tried;
        }
    }
    return from_lane0(item, lane);
}

template <int G>
__device__ __forceinline__ void load_half_vec(const __half* p, float (&v)[G]) {
    if constexpr (G == 8) {
        uint4 r = *reinterpret_cast<const uint4*>(p);
        const __half2* hp = reinterpret_cast<const __half2*>(&r);
#pragma unroll
        for (int j = 0; j < 4; ++j) { float2 f = __half22float2(hp[j]); v[2 * j] = f.x; v[2 * j + 1] = f.y; }
    } else if constexpr (G == 4) {
        uint2 r = *reinterpret_cast<const uint2*>(p);
        const __half2* hp = reinterpret_cast<const __half2*>(&r);
#pragma unroll
        for (int j = 0; j < 2; ++j) { float2 f = __half22float2(hp[j]); v[2 * j] = f.x; v[2 * j + 1] = f.y; }
    } else if constexpr (G == 2) {
        float2 f = __half22float2(*reinterpret_cast<const __half2*>(p));
        v[0] = f.x; v[1] = f.y;
    } else {
        v[0] = __half2float(*p);
    }
}

// The same load without the conversion (the bits wait in (G+1)/2 registers), and the conversion.
template <int G>
__device__ __forceinline__ void load_half_raw(const __half* p, uint32_t (&raw)[(G + 1) / 2]) {
    if constexpr (G == 8) {
        const uint4 r = *reinterpret_cast<const uint4*>(p);
        raw[0] = r.x; raw[1] = r.y; raw[2] = r.z; raw[3] = r.w;
    } else if constexpr (G == 4) {
        const uint2 r = *reinterpret_cast<const uint2*>(p);
        raw[0] = r.x; raw[1] = r.y;
    } else if constexpr (G == 2) {
        raw[0] = *reinterpret_cast<const uint32_t*>(p);
    } else {
        raw[0] = (uint32_t)__half_as_ushort(*p);
    }
}
template <int G>
__device__ __forceinline__ void half_raw_to_float(const uint32_t (&raw)[(G + 1) / 2], float (&v)[G]) {
    if constexpr (G == 1) {
        v[0] = __half2float(__ushort_as_half((unsigned short)raw[0]));
    } else {
#pragma unroll
        for (int j = 0; j < G / 2; ++j) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&raw[j]));
            v[2 * j] = f.x; v[2 * j + 1] = f.y;
        }
    }
}

template <int G>
__device__ __forceinline__ void store_vec(void* base, long long elem, const float (&v)[G], int out_f16) {
    if (out_f16) {
        __half* p = reinterpret_cast<__half*>(base) + elem;
        if constexpr (G == 1) { *p = __float2half_rn(v[0]); }
        else {
            __half2 t[G / 2];
#pragma unroll
            for (int j = 0; j < G / 2; ++j) t[j] = __floats2half2_rn(v[2 * j], v[2 * j + 1]);
            if constexpr (G == 8) *reinterpret_cast<uint4*>(p) = *reinterpret_cast<uint4*>(t);
            else if constexpr (G == 4) *reinterpret_cast<uint2*>(p) = *reinterpret_cast<uint2*>(t);
            else *reinterpret_cast<__half2*>(p) = t[0];
        }
    } else {
        float* p = reinterpret_cast<float*>(base) + elem;
        if constexpr (G >= 4) {
#pragma unroll
            for (int j = 0; j < G / 4; ++j)
                reinterpret_cast<float4*>(p)[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        } else if constexpr (G == 2) { *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]); }
        else { *p = v[0]; }
    }
}

struct Item {
    int t, s, c;        // table, session, chunk
    int p0, P;          // first position, positions in the chunk (0: no such chunk)
    long long slot;
};

__device__ __forceinline__ Item bulk_item(const CodecArgs& a, unsigned item, int t_first = 0) {
    Item it;
    const unsigned per_table = (unsigned)a.S * (unsigned)a.chunks;
    it.t = t_first + (int)(item / per_table);
    unsigned r = item % per_table;
    it.s = (int)(r / a.chunks);
    it.c = (int)(r % a.chunks);
    const int Wt = 2 * a.sh.L * a.sh.H;
    it.slot = ((long long)it.s * Wt + it.t) * a.st.max_chunks + it.c;
    int b = a.pos_begin ? a.pos_begin[it.s] : 0, e = a.pos_end ? a.pos_end[it.s] : a.n;
    b = max(b, 0); e = min(e, a.n);
    long long p0 = (long long)b + (long long)it.c * a.sh.chunk_pos;
    it.p0 = (int)min(p0, (long long)a.n);
    it.P = p0 < e ? min(a.sh.chunk_pos, e - (int)p0) : 0;
    return it;
}

// Encoders rewrite the whole index of the launch's tables: the entries behind the chunks that a session of
// this call can have, by the whole grid.
__device__ __forceinline__ void clear_unused_slots(const CodecArgs& a, int t_first, int n_tables) {
    const int room = a.st.max_chunks - a.chunks, Wt = 2 * a.sh.L * a.sh.H;
    const long long total = (long long)a.S * n_tables * room;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const long long stream = i / room;
        const long long slot = (stream / n_tables * Wt + t_first + stream % n_tables) * a.st.max_chunks + a.chunks + i % room;
        a.st.chunk_offset[slot] = 0; a.st.chunk_bytes[slot] = 0;
    }
}

__device__ __forceinline__ long long kv_elem(const KvView& v, int t, int H, int s, int pos) {
    int layer = t / (2 * H), kv = (t / H) & 1, head = t % H;
    return layer * v.sl + kv * v.skv + s * v.ss + head * v.sh + (long long)pos * v.sp;
}

// Copies n 16-bit words to a 16-byte aligned destination from a 2-byte aligned source, 16 bytes a lane
// and step (`lane` of `lanes` threads; two-byte copies cost the tail of a chunk as much as a quarter of
// its coding).  The source is read in aligned 32-bit words, up to two bytes before and behind the
// range: the staging areas have that room.
__device__ __forceinline__ void copy_words(uint8_t* dst, const uint16_t* src, int n, int lane, int lanes) {
    const uint32_t* s4 = reinterpret_cast<const uint32_t*>(reinterpret_cast<uintptr_t>(src) & ~(uintptr_t)3);
    const uint32_t sh = (reinterpret_cast<uintptr_t>(src) & 2) ? 16u : 0u;
    const int n16 = n >> 3;                                   // whole 16-byte pieces
#pragma unroll 2
    for (int i = lane; i < n16; i += lanes) {
        uint32_t w[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) w[j] = __ldcg(s4 + 4 * i + j);
        reinterpret_cast<uint4*>(dst)[i] = make_uint4(__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh),
                                                      __funnelshift_r(w[2], w[3], sh), __funnelshift_r(w[3], w[4], sh));
    }
    for (int i = 8 * n16 + lane; i < n; i += lanes) reinterpret_cast<uint16_t*>(dst)[i] = __ldcg(src + i);
}

// Reserves a finished chunk's place: writes its states, index entry and counters; returns where its words
// go, or null if they must not be written.  One warp.
__device__ __forceinline__ uint8_t* reserve_chunk(const CodecArgs& a, long long slot, uint32_t x, int n_words, int lane, int P,
                                                  unsigned n_escapes, int n_skipped) {
    const unsigned nbytes = 128u + 2u * (unsigned)n_words;
    unsigned long long off = 0;
    if (lane == 0) {
        off = atomicAdd(a.st.total_bytes, (unsigned long long)((nbytes + 15u) & ~15u));
        atomicAdd(&a.counters->payload_bytes, (unsigned long long)nbytes);
        atomicAdd(&a.counters->n_chunks, 1ull);
        atomicAdd(&a.counters->coded_vectors, (unsigned long long)P);
        if (n_skipped) atomicAdd(&a.counters->skipped_vectors, (unsigned long long)n_skipped);
        if (n_escapes) atomicAdd(&a.counters->n_escapes, (unsigned long long)n_escapes);
    }
    off = __shfl_sync(kFull, off, 0);
    const bool fits = off + nbytes <= a.st.capacity;
    const bool aligned = (off & 15ull) == 0;             // the caller's byte cursor must be a multiple of 16
    if (lane == 0) {
        a.st.chunk_offset[slot] = off;
        a.st.chunk_bytes[slot] = nbytes;
        if (!fits) atomicOr(a.status, kStCapacity);
        if (!aligned) atomicOr(a.status, kStCursor);
    }
    if (!fits || !aligned) return nullptr;
    uint8_t* dst = a.st.payload + off;
    reinterpret_cast<uint32_t*>(dst)[lane] = x;
    return dst + 128;
}

// Finishes an encoded chunk whose words one warp has staged at stage[wp, cap_words).
__device__ __forceinline__ void commit_chunk(const CodecArgs& a, long long slot, uint32_t x, const uint16_t* stage,
                                             int wp, int cap_words, int lane, int P, unsigned n_escapes, int n_skipped = 0) {
    __syncwarp();
    uint8_t* dst = reserve_chunk(a, slot, x, cap_words - wp, lane, P, n_escapes, n_skipped);
    if (dst) copy_words(dst, stage + wp, cap_words - wp, lane, 32);
}

// Quantiser decision in binary32: sym = rint((kv - mu) * fl(1/delta)), clamped to +-2^30.
__device__ __forceinline__ int quantise(float kv, float mu, float inv_delta) {
    const float n = __fmul_rn(__fsub_rn(kv, mu), inv_delta);
    return __float2int_rn(fminf(fmaxf(n, -(float)kSymLimit), (float)kSymLimit));   // the limits are whole numbers: as if rounded first
}

extern __shared__ __align__(16) int2 g_pair_smem[];   // per warp: two slots of Kp entries

// Prediction read from the dense variant's buffers: mu [row][tables of the launch * D] and the variance
// term s1 [row][tables of the launch] (sum_v p_v ||T_v||^2 / d); sigma2 = max(0, s1 - ||mu||^2 / d).
template <int D>
__device__ __forceinline__ void dense_fetch(const CodecArgs& a, long long row, int t_local, int c0,
                                            float (&m)[Geo<D>::G], float& s1) {
    constexpr int G = Geo<D>::G;
    const float* mp = a.mu_dense + row * a.mu_ld + (long long)t_local * D + c0;
#pragma unroll
    for (int g = 0; g < G; ++g) m[g] = __ldg(mp + g);
    s1 = __ldg(a.s1_dense + row * a.s1_ld + t_local);
}
template <int D>
__device__ __forceinline__ void dense_finish(const CodecArgs& a, int t_local, int c0, float inv_d, const float (&m)[Geo<D>::G],
                                             float s1, float (&mu)[Geo<D>::G], float& sigma2) {
    constexpr int G = Geo<D>::G;
#pragma unroll
    for (int g = 0; g < G; ++g) mu[g] = m[g];
    if (a.mu_bias) {
#pragma unroll
        for (int g = 0; g < G; ++g) mu[g] = __fadd_rn(mu[g], __half2float(a.mu_bias[t_local * D + c0 + g]));
    }
    const float s2 = warp_norm2<G>(mu);
    sigma2 = fmaxf(0.f, s1 - s2 * inv_d);
}

enum { kSrcGather = 0, kSrcOpen = 1, kSrcDense = 2 };

template <class F>
inline cudaError_t dispatch_d(int d, F&& f) {
    switch (d) {
        case 32: return f(std::integral_constant<int, 32>{});
        case 64: return f(std::integral_constant<int, 64>{});
        case 128: return f(std::integral_constant<int, 128>{});
        case 256: return f(std::integral_constant<int, 256>{});
    }
    return cudaErrorInvalidValue;
}

// Dynamic shared memory that the kernels are let take: K = 1024 is the most pairs, 144 KB with the slots of a
// block of eight warps; 34 KB of tables are static.  The limit belongs to the function, for all contexts and
// threads of the process, so it is set to this value always: no thread's launch falls between another's
// set and launch.
constexpr size_t kMostSmem = 160 * 1024;
template <class... P>
cudaError_t allow_smem(void (*kern)(P...), size_t bytes) {
    return bytes > kMostSmem ? cudaErrorInvalidValue : cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMostSmem);
}

}  // namespace
}  // namespace plc
