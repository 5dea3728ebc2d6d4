// Shared definitions of the libplc CUDA translation units (sm_100a only).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "plc.h"

namespace plc {

constexpr int kProbBits = 15;
constexpr uint32_t kProbM = 1u << kProbBits;
constexpr uint32_t kRansL = 1u << 16;
constexpr int kNumSym = 64;        // zigzag(hi), hi in [-31,31] -> 0..62; 63 = escape
constexpr int kEsc = 63;
constexpr int kHiMax = 31;
constexpr int kQMin = -24;
constexpr int kQMax = 135;
constexpr int kNumTables = 40;     // table id qp in [-24, 15]
constexpr int kSymLimit = 1 << 30;
constexpr uint32_t kFull = 0xffffffffu;

// Bits of the device status word.
constexpr uint32_t kStCapacity = 1u, kStCorrupt = 2u, kStBadClass = 4u, kStTimeout = 8u, kStCursor = 16u;

// Device counters (plc_stats).
struct Counters {
    unsigned long long payload_bytes, n_chunks, n_escapes, coded_vectors, skipped_vectors;
    double ideal_bits;     // code length under the coder's model (only counted on request)
};

// Frequency-table entry used by the encoder: rcp = floor(2^32 / f) (2^32-1 for f = 1),
// fc = f | (c << 16).
struct EncEntry {
    uint32_t rcp, fc;
};

// Two 32-bit constants per table id: theta = round(2^32 exp(-sqrt2/s')), rho = round(2^32
// exp(-sqrt2/(2 s'))), s' = 2^(qp/8).  Literal so that encoder and decoder builds agree bit for bit.
__host__ __device__ inline void table_constants(int qp, uint32_t& theta, uint32_t& rho) {
    constexpr uint32_t kC[kNumTables][2] = {
        {52418u, 15004422u},         {134053u, 23994893u},        {317125u, 36905875u},
        {698470u, 54771407u},        {1440801u, 78665070u},       {2798733u, 109637892u},
        {5145013u, 148652826u},      {8992185u, 196522626u},      {15004422u, 253857248u},
        {23994893u, 321025356u},     {36905875u, 398132550u},     {54771407u, 485016909u},
        {78665070u, 581260615u},     {109637892u, 686215099u},    {148652826u, 799036310u},
        {196522626u, 918726429u},    {253857248u, 1044178424u},   {321025356u, 1174220339u},
        {398132550u, 1307656790u},   {485016909u, 1443305845u},   {581260615u, 1580030169u},
        {686215099u, 1716761896u},   {799036310u, 1852521207u},   {918726429u, 1986428948u},
        {1044178424u, 2117713904u},  {1174220339u, 2245715466u},  {1307656790u, 2369882518u},
        {1443305845u, 2489769347u},  {1580030169u, 2605029347u},  {1716761896u, 2715407188u},
        {1852521207u, 2820730047u},  {1986428948u, 2920898384u},  {2117713904u, 3015876649u},
        {2245715466u, 3105684222u},  {2369882518u, 3190386796u},  {2489769347u, 3270088366u},
        {2605029347u, 3344923893u},  {2715407188u, 3415052718u},  {2820730047u, 3480652712u},
        {2920898384u, 3541915165u}};
    theta = kC[qp - kQMin][0];
    rho = kC[qp - kQMin][1];
}

// Discretised Laplace frequencies of table qp, integer recurrence:
// G0 = 2^32, G1 = rho, G(k+1) = (Gk theta) >> 32; f(0) = (G0-G1) >> 17, f(+-k) = (Gk-Gk+1) >> 18,
// f(ESC) = G32 >> 17, each at least 1; f(0) absorbs the difference to 2^15.
__host__ __device__ inline void build_freqs(int qp, uint32_t* f /*[64]*/) {
    uint32_t theta, rho;
    table_constants(qp, theta, rho);
    unsigned long long g = 1ull << 32, gn = rho;
    unsigned long long m = (g - gn) >> 17;
    f[0] = m < 1 ? 1u : (uint32_t)m;
    g = gn;
    for (int k = 1; k <= kHiMax; ++k) {
        gn = (g * (unsigned long long)theta) >> 32;
        m = (g - gn) >> 18;
        uint32_t fk = m < 1 ? 1u : (uint32_t)m;
        f[2 * k - 1] = fk;
        f[2 * k] = fk;
        g = gn;
    }
    m = g >> 17;
    f[kEsc] = m < 1 ? 1u : (uint32_t)m;
    long long sum = 0;
    for (int i = 0; i < kNumSym; ++i) sum += f[i];
    f[0] = (uint32_t)((long long)f[0] + ((long long)kProbM - sum));
}

// Scale class -> (number of bit planes s, table id qp).
__host__ __device__ inline void class_params(int q, int& s, int& qp) {
    if (q < 16) { s = 0; qp = q; }
    else { s = (q >> 3) - 1; qp = 8 + (q & 7); }
}

#ifdef __CUDACC__
// Programmatic dependent launch: a kernel launched with `chained` set may start before the kernel ahead of
// it in the stream has finished; it calls chain_wait before it touches anything another kernel wrote or
// still reads, and chain_next as soon as its own successor may be started.  What it saves is the launch
// gap between short kernels (1 to 3 us).  What it can cost: blocks that become resident beside those of the
// kernel ahead take over their SM's division of L1 and shared memory for as long as they run (the coder
// behind a top-K of many rows, which holds up to 213 KB of shared memory an SM: 64 sessions' tails, rows from
// HBM, 18.3 -> 29.0 ms), and crowd on the SMs that are free first (128 chunks, a block each: 355 -> 447 us).
// A chained kernel is resident while the kernel ahead writes, so what that kernel (or the caller's own, whose
// logits a chained top-K reads) may write is read with ordinary loads: the non-coherent path (__ldg) asks for
// data that does not change while the kernel lives.  T, row norms and coder tables may take it, and payload
// words and records, since no kernel is chained to an encoder or decoder.
// So a kernel is chained only where neither can happen: see launch_coop and plc_append_step's launches.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <class... P, class... A>
inline cudaError_t launch_kernel(void (*kern)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, bool chained, unsigned cluster,
                                 A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2]{};
    cfg.attrs = at;
    if (chained) {
        at[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        at[cfg.numAttrs].val.clusterDim.x = cluster;
        at[cfg.numAttrs].val.clusterDim.y = at[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// q = clamp(round(4 log2 v), kQMin, kQMax), decided on the binary32 exponent and four mantissa
// thresholds 2^((2i+1)/8); v <= 0 -> kQMin.
__device__ __forceinline__ int class_from_v(float v) {
    if (!(v > 0.0f)) return kQMin;
    uint32_t b = __float_as_uint(v);
    int e = (int)(b >> 23);
    if (e == 255) return kQMax;
    float m;
    if (e == 0) {                      // subnormal: far below the smallest class
        return kQMin;
    }
    m = __uint_as_float((b & 0x007fffffu) | 0x3f800000u);   // [1,2)
    int q = 4 * (e - 127);
    q += (m >= 1.09050773f) + (m >= 1.29683955f) + (m >= 1.54221083f) + (m >= 1.83400809f);
    return min(max(q, kQMin), kQMax);
}

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Packed pairs of binary32 (sm_100 f32x2 instructions) in register pairs that stay packed across a loop; each
// half is an IEEE operation, so the result equals two scalar ones.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1,%2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) {
    asm("mov.b64 {%0,%1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

#endif

// SMs of the current device.
inline int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 148;
    return sms;
}

// Host-side launch counter shared by all translation units.
void count_launch(int n = 1);

constexpr int kTicketWords = 1024;               // one counter per work queue (at most one queue per SM)

// Internal launchers (one per .cu file).
struct TopkArgs {
    const __half* logits; const int32_t* tokens; int64_t N; int V, K;
    int2* pairs;            // [N][Kp], or null: see put_pair; entries K..Kp-1 get candidate 0 with weight 0
    int Kp, pair_rows, pair_mul;   // log2 of the rows a warp-wide load fetches; bytes of a table row (1: pairs hold indices)
    int32_t* idx; float* w; float* lse; float* zk; float* logp2;   // optional user outputs
    // Adaptive step (needs tokens): step_exp[row] = b0 - b_i, bits_out[row] = b_i (both optional).
    int* step_exp; int* bits_out; int b0, extra; float hbar;
    // Rows are skipped (nothing written) when pos ranges are given and the row is outside them.
    int n_per_session; const int32_t* pos_begin; const int32_t* pos_end;
    int parts;              // parts of a row where its sum must not depend on the call (set by the launcher)
    unsigned int* tickets;  // kTicketWords work counters that the launch zeroes for the kernel behind it, or null
    bool chained;           // where rows are few, the launch may start while the kernel ahead of it ends
};
// *few_blocks: the blocks launched where rows are few (several warps a row, little shared memory; or at most a
// block an SM), else 0.
cudaError_t launch_topk(const TopkArgs& a, cudaStream_t st, int* few_blocks);

cudaError_t launch_prefix_dedup(const int32_t* tokens, const int32_t* lens, const float* logp2, int S, int64_t stride,
                                int32_t* lcp, float* dT, int32_t* parent, int32_t* shared_len, cudaStream_t st);

cudaError_t launch_prefix_clusters(const int32_t* lcp, const float* dT, int S, float delta, int32_t* cluster,
                                   int32_t* centroid, int32_t* begin, cudaStream_t st);

constexpr int kZeroOff = -1000000;

struct CodecShape {
    int L, H, d, V, K, Kp, chunk_pos, out_dtype;   // Kp: K rounded up to twice the rows one warp-wide load fetches
    float delta, sigma_floor;
    float inv_delta, inv_delta2;   // fl(1/delta), fl(1/(delta*delta)), rounded once on the host
    int zero_q;                    // zero-rate rule (Thm. 3): positions of class <= zero_q carry no symbols (kZeroOff = never)
};

struct KvView {
    void* base; int64_t sl, skv, ss, sh, sp;
};

struct StreamsDev {
    uint8_t* payload; unsigned long long capacity; unsigned long long* chunk_offset; uint32_t* chunk_bytes;
    unsigned long long* total_bytes; int max_chunks;
};

struct DebugDev {
    int32_t* sym; int32_t* q; float* mu;
    int ideal;             // non-zero: add every coded component's model code length to Counters::ideal_bits
};

struct CoderTables;                                // plc_coder.cuh

struct CodecArgs {
    CodecShape sh;
    const CoderTables* tables;                     // frequency tables of the coder
    const __half* T; const float* rownorm2;        // [tables][V][d], [tables][V]
    const float* norms_by_row;                     // [V][tables], for launch_variance
    float* s1;                                     // [S*n][tables] variance terms where they were formed ahead (launch_variance), or null
    const int2* pairs;                             // [S*n][Kp] (written by the top-K kernels, put_pair)
    bool pair_index;                               // pairs hold row indices instead of byte offsets (tables of 4 GB or more)
    bool finite;                                   // T holds neither infinities nor NaN
    const int* step_exp;                           // [S*n] adaptive step exponent, or null
    KvView kv;                                     // encode: input f16; decode: output
    int S, n; const int32_t* pos_begin; const int32_t* pos_end;
    int chunks;                                    // chunks a session of the call can have, ceil(n / chunk_pos): the unit of work; st.max_chunks is the room of the index
    StreamsDev st; DebugDev dbg;
    uint16_t* staging; unsigned long long staging_words_per_warp;   // encoder scratch
    unsigned int* ticket;                          // kTicketWords work counters (zeroed by the top-K launch, or by the launcher where none precedes)
    int behind;                                    // blocks of the top-K launch ahead that this one may be chained to, or 0
    int sched_nq, sched_g;                         // gather kernels: work queues, SMs that share one (set by the launcher)
    unsigned int* status; Counters* counters;
    // dense variant: prediction read from buffers; one launch covers tables [dense_t0, dense_t0 + dense_nt)
    const float* mu_dense; const float* s1_dense; long long mu_ld, s1_ld; int dense_t0, dense_nt;
    const __half* mu_bias;                         // optional [dense_nt][d] f16 added to mu (linear predictor's c), or null
    // append path: symbols come from / go to the open chunk
    int32_t* open_sym; int32_t* open_q; int open_slot; int open_count; int chunk_index;
    unsigned open_first, open_items;               // seal launch: the (table, session) items [open_first, open_first + open_items)
};
int codec_grid_warps(int device);
// Work-queue layout a gather launch over n_tables tables would use: nq queues, g SMs per queue.
void codec_schedule(const CodecArgs& a, int n_tables, int* nq, int* g);

// Rotated fixed-rate quantiser (Prop. 3 step 3): records of 1 + (d/32)*bits words per (stream, position),
// record of (session s, table t, position i) at word ((s*W + t)*n + i) * rec_words.
struct RotqArgs {
    int bits;
    uint32_t sign_bits[8];      // bit j set: component j is negated before and after the transform
    uint32_t* records;
    int rec_words;
};
cudaError_t launch_rotq(const CodecArgs& a, const RotqArgs& r, bool encode, cudaStream_t st);

// Dense (full-vocabulary) prediction, a group of layers at a time.
struct DenseShape {
    long long rows;        // S * n positions
    int V, d, tables;      // tables = 2 * H of one layer
    int ldv;               // V rounded up to 64 (row pitch of P, Tb and Nb, in elements)
    int ncols;             // tables * d
    int nt_all;            // L * tables (one variance column per layer and table)
    int group;             // layers per contraction
    bool resident;         // the context keeps the transposed bf16 table of every layer
};
int layers_per_group(int L, long long rows, int ncols);
size_t dense_scratch_bytes(const DenseShape& sh, size_t* off /*[4]: P, Tb, mu, s1*/);
size_t dense_model_bytes(const DenseShape& sh, size_t* off /*[2]: Nb_all, Tb_all*/);
cudaError_t dense_prepare(const __half* T, const DenseShape& sh, uint8_t* model, const size_t* moff, cudaStream_t st);
cudaError_t dense_softmax(const __half* logits, const DenseShape& sh, uint8_t* scratch, const size_t* off, cudaStream_t st);
cudaError_t dense_layers(const __half* T, int l0, int nl, const DenseShape& sh, const uint8_t* model, const size_t* moff, uint8_t* scratch,
                         const size_t* off, unsigned int* status, cudaStream_t st, cudaEvent_t ev0, cudaEvent_t ev1);   // events bracket the contraction
// Linear-embedding predictor (Sec. 7.1).
struct LinearShape {
    long long rows;
    int V, d, dm, tables, L;   // tables = 2*H per layer, dm = d_model (multiple of 64)
    int ldv;                   // V rounded up to 64
    int ncols;                 // tables*d
    int nt_all;                // L*tables
    int group;                 // layers per contraction
    bool resident;             // the context keeps A as bf16
};
size_t linear_model_bytes(const LinearShape& sh, size_t* off /*[3]*/);
size_t linear_scratch_bytes(const LinearShape& sh, size_t* off /*[5]*/);
cudaError_t linear_prepare(const __half* E, const __half* A, const __half* c, const LinearShape& sh, uint8_t* model,
                           const size_t* moff, unsigned int* status, cudaStream_t st);
cudaError_t linear_begin(const __half* logits, const LinearShape& sh, const uint8_t* model, const size_t* moff,
                         uint8_t* scratch, const size_t* off, unsigned int* status, cudaStream_t st);
cudaError_t linear_layers(const __half* A, int l0, int nl, const LinearShape& sh, const uint8_t* model, const size_t* moff, uint8_t* scratch,
                          const size_t* off, unsigned int* status, cudaStream_t st, cudaEvent_t ev0, cudaEvent_t ev1);
// Sets *not_finite where a row holds an infinity or NaN.
cudaError_t launch_rownorm(const __half* T, float* out, long long rows, int d, unsigned int* not_finite, cudaStream_t st);
cudaError_t launch_norms_by_row(const float* norms, float* by_row, int V, int tables, cudaStream_t st);
cudaError_t launch_variance(const CodecArgs& a, cudaStream_t st);            // fills a.s1 for the pairs
cudaError_t launch_encode(const CodecArgs& a, cudaStream_t st);
cudaError_t launch_decode(const CodecArgs& a, cudaStream_t st);
cudaError_t launch_coop(const CodecArgs& a, bool encode, cudaStream_t st);   // a block per chunk; queues set, tickets zeroed
cudaError_t launch_append_quantise(const CodecArgs& a, cudaStream_t st);   // predict + quantise into the open chunk
cudaError_t launch_append_seal(const CodecArgs& a, cudaStream_t st);       // code the open chunk

}  // namespace plc
