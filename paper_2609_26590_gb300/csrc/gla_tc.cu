// gla_tc.cu -- tensor-core chunkwise schedule of the GTR token mixer for sm_103a.
//
// Method (Sec. 3.3, Eq. chunk_boundary_main and the chunk-output formula after
// it; chunk size C = 64 as in App. C.3).  For chunk c of a (b, h) sequence, with
// in-chunk scan position r and A_r = sum_{m<=r} g_m (per key channel):
//   o_r      = (q_r . e^{A_r}) S_[c] + sum_{j<=r} (sum_i q_ri k_ji e^{A_ri - A_ji}) v_j
//   U_c      = sum_r (k_r . e^{A_last - A_r})^T v_r,   d_c = e^{A_last}
//   S_[c+1]  = Diag(d_c) S_[c] + U_c
// A persistent CTA per SM walks all chunks of its (b, h) sequences as one stream
// (single pass: q, k, v, g are read once, o and S_final written once; S stays on
// chip between chunks, and the pipeline does not drain between sequences).
//
// Per chunk, tensor-core products (tcgen05.mma, fp32 accumulators in TMEM):
//   A = L G          in-chunk cumulative log-decay: L is the 64x64 triangle of
//                    ones in scan order, G the gate tile as loaded (exact products)
//   P = Q^ K^^T      intra-chunk scores with e^{A_r - A_j} split at the mid-chunk
//                    reference: Q^ = q e^{A_r - A_mid}, K^ = k e^{A_mid - A_j}
//   U = Kbar^T V     chunk summary, Kbar = k e^{A_last - A}
//   O = Qtil S_[c] + P V   outputs, Qtil = q e^{A}
// The split factors of P lie within 2^{+-M}, M = max_i max(-A_mid, A_mid - A_last)
// (log2 units).  M <= 8 ("fp16 mode"): Q^, K^ are fp16 and serve all products,
// because the per-channel constants c1 = e^{A_mid}, c2 = e^{A_last - A_mid} fold
// into the state: Qtil S = Q^ (Diag(c1) S) and Kbar^T V = Diag(c2) K^^T V.
// M <= 100 ("tf32 mode"): Q^, K^ are tf32 (fp32 range) for P, and Qtil, Kbar are
// written as fp16 operands.  Larger M or non-finite gates ("exact mode"): the
// chunk's log-decays and scores are computed exactly by CUDA cores.
//
// Memory: each chunk owns a 32 KB stage slot (q, k, v, g tiles) from its TMA
// load until its output product completes; the derived fp16 operands are
// written in place (Q^ or Qtil over q, K^ or Kbar over k, the masked scores P
// over g, bf16 v converted to fp16 in place), so four chunks can be in flight.
// Only the tf32 score operands use separate buffers, one per gen warpgroup, so
// that tf32-mode chunks of the two groups never wait for each other.  Row orders
// load one 64-row TMA box per tensor and chunk; column orders one im2col load per
// tensor (a map whose fastest spatial dimension is the grid row, so 64 pixels run
// down a column and on into the next).  Chunks that reach past either end of the
// sequence load one box per column segment instead, of the segment's exact height (a
// tensor map per height), and zero-fill boxes for the rows outside.  The scan
// permutation lives in the load coordinates and in the addresses of the output stores.
//
// Warp roles (512 threads, one CTA per SM; four warps per SM sub-partition, so a
// thread keeps 128 registers).  All roles share the SM's instruction cache, so few
// roles with small loops:
//   warp 0       TMA producer.
//   warp 1       TMEM allocator and issuer of A(c) = L G.
//   warps 2-5    gen warpgroup 0 (even chunks): reads A, builds the operands of its
//                chunk, then masks the chunk's scores P into fp16.
//   warps 6-9    gen warpgroup 1 (odd chunks).
//   warps 10-13  epi: carries the fp32 state S in registers, writes Diag(c1) S,
//                and stores each chunk's outputs at the tokens' spatial positions
//                (GENOUT launches: the gen warpgroup that built the chunk stores them).
//   warp 14      issuer of P(c) and U(c).
//   warp 15      issuer of O(c).
// (Two key halves: warps 0-3 producer, A, P/U and O issuers, 4-7 and 8-11 gen, 12-15 epi.)
// Each issuer waits only for the inputs of its own product, so the issue overhead
// of one product does not hold up the others.
// A warp reads the TMEM lanes of sub-partition (warp % 4); an M = 64 accumulator
// keeps rows 16q..16q+15 in lanes 32q..32q+15, and each thread takes one row and
// 32 of its 64 columns.
//
// Few, long sequences are split into segments (MODE kSummary computes each
// segment's end state from zero and its total decay, MODE kSplitFull starts every
// segment from the fold of the earlier ones); the last segment may run past the
// sequence over all-zero padding chunks, which leave the state unchanged.  When the
// units outnumber the SMs unevenly (MODE kBalanced), every CTA takes an equal
// contiguous range of the units' chunks: the head of the unit its range ends in comes
// first and hands its end state to the next CTA through global memory, the tail of
// the unit its range starts in comes last, from the state the CTA before handed over.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <atomic>
#include <chrono>
#include <cstdlib>
#include <cstring>
#include <list>
#include <mutex>
#include <type_traits>

#include "f32x2.cuh"
#include "fastdiv.cuh"
#include "gla_internal.h"
#include "tc_ptx.cuh"

namespace gtr {

__device__ unsigned int g_device_status;

namespace {

using namespace ptx;

constexpr int kC = 64;                    // chunk length
constexpr int kD = 64;                    // Dk = Dv handled by this kernel
constexpr int kSlots = 4;                 // stage slots (chunks in flight)
constexpr int kTile16 = kC * kD * 2;      // 64 x 64 16-bit tile (SW128, 128-byte rows)
constexpr int kTile32 = kC * kD * 4;      // 64 x 64 fp32 tile (two 32-column K-blocks)
constexpr int kThreads = 512;
constexpr int kHeights = 15;              // TMA box heights 1 .. 7, then 8, 16, ..., 64
// Rows of the TMA box of height index hi (one tensor map per height).
__host__ __device__ constexpr int box_height(int hi) { return hi < 7 ? hi + 1 : 8 * (hi - 6); }
constexpr uint64_t kWaitLimitNs = 1000000000ull;  // bounded waits give up after 1 s
// what a chunk of a summary pass may take, on top of that, for the output pass that waits for it: ten times
// what the slowest ones (all scores exact) take
constexpr uint64_t kSummaryChunkNs = 100000ull;
constexpr float kLog2e = 1.4426950408889634f;
// Gates below this (log2) act as it: 2^-128 is 0 (flushed) as any smaller decay is, and a chunk's prefix stays
// above -8,192, whose last bit of 2^-10 the decays of the keys after a channel's last zero gate keep.  (With
// gates clamped at -1e4 a few zero gates a channel left the prefix 2^-5 and the outputs 4e-3 off.)
constexpr float kGateMinLog2 = -128.0f;
constexpr float kMaxRefF16 = 8.0f;        // fp16 score operands: factors within 2^{+-8}
constexpr float kMaxRefTF32 = 100.0f;     // tf32 score operands: factors within 2^{+-100}

enum : uint32_t { kModeF16 = 0, kModeTF32 = 1, kModeExact = 2 };
// Kernel passes: kFull (sequences whole, dealt round-robin), kSplitFull (outputs of
// segments that start from the fold of the earlier segments' summaries), kSummary (the
// summaries), kBalanced (equal contiguous chunk ranges per CTA, the state of a unit cut
// by a range boundary handed from one CTA to the next; one key half).
enum : int { kFull = 0, kSplitFull = 1, kSummary = 2, kBalanced = 3 };
constexpr int kMinSegChunks = 2;          // a split segment keeps at least this many chunks
constexpr int kMaxUnsplitChunks = 5;      // shorter sequences are never split
constexpr uint32_t kBarSetup = 4;         // named barrier: set-up done
constexpr uint32_t kBarSin = 5;           // named barrier (two key halves): epi read the folded start state

// Shared-memory map (byte offsets from a 1024-aligned base).
constexpr int kSlotBytes = 4 * kTile16;                        // q @0, k @8K, v @16K, g @24K
constexpr int kQ = 0, kK = kTile16, kV = 2 * kTile16, kG = 3 * kTile16;
constexpr int kOffSlot = 0;
constexpr int kOffOp = kOffSlot + kSlots * kSlotBytes;         // per gen group g @32K g: tf32 Q^ @0, K^ @16K
constexpr int kOffS = kOffOp + 4 * kTile32;                    // 2 x S'_[c] (fp16, MN-major)
constexpr int kOffL = kOffS + 2 * kTile16;                     // triangle of ones
constexpr int kRank = 16;                                      // rank r of the gate's low-rank projection
constexpr int kW2Bytes = kRank * kD * 2;                       // a head's W2 block: r x 64 channels, 16-bit
constexpr int kOffW2 = kOffL + kTile16;                        // gate producer: 2 x W2 (by unit parity)
constexpr int kRefFloats = 4 * kD;                             // -A_mid, -A_last (log2), c1, c2
constexpr int kOffRef = kOffW2 + 2 * kW2Bytes;                 // per slot
constexpr int kOffDecay = kOffRef + kSlots * kRefFloats * 4;   // per slot, 64 fp32
constexpr int kOffMode = kOffDecay + kSlots * kD * 4;          // per slot u32 mode; 2 x 2 fp32 maxima
constexpr int kOffBar = kOffMode + 64;
// the start state's fold (one key half): summaries whose decay products fit the S' buffers; row pitch
constexpr int kFoldBatch = 32, kFoldPitch = 68;
static_assert(kSlots >= 4 && 2 * kSlotBytes >= 4 * kD * kD * 4 && kFoldBatch * kD * 4 <= 2 * kTile16, "the fold's ring and coefficients");
constexpr int kNumBars = 40;
constexpr int kOffMisc = kOffBar + kNumBars * 8;               // tmem base, abort flag
constexpr int kSmemBytes = kOffMisc + 64 + 1024;               // + alignment slack
static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");

enum {
    BAR_FULL = 0,                      // [kSlots] TMA -> issuer (A)
    BAR_EMPTY = BAR_FULL + kSlots,     // [kSlots] U(c) and O(c) done (two commits) -> producer
    BAR_REFS = BAR_EMPTY + kSlots,     // [kSlots] gen -> epi: chunk constants and mode
    BAR_AFULL = BAR_REFS + kSlots,     // [2] A done -> gen
    BAR_PURDY = BAR_AFULL + 2,         // [2] P/U(c) may go: gen(c) operands in smem and A(c) read
                                       //     (4 arrivals) + epi drained U(c-2) (4 arrivals)
    BAR_PFULL = BAR_PURDY + 2,         // [2] P done -> gen
    BAR_UFULL = BAR_PFULL + 2,         // [2] U done -> epi
    BAR_ORDY = BAR_UFULL + 2,          // [2] O(c) may go: gen(c) masked P in smem and TMEM P read
                                       //     (4) + epi wrote Diag(c1) S_[c] and read O(c-2) (4)
    BAR_OFULL = BAR_ORDY + 2,          // [2] O of a virtual chunk done -> epi
    BAR_ZFULL = BAR_OFULL + 2,         // [2] gate producer: Z = a W2 done -> gen
    BAR_GRDY = BAR_ZFULL + 2,          // [2] gate producer: gates G written by the gen group (4) -> A issuer
    BAR_DONE = BAR_GRDY + 2,           // every MMA completed (teardown)
    BAR_SIN = BAR_DONE + 1,            // kSplitFull: the epi folded the start state (4) -> producer
    BAR_GFULL = BAR_SIN + 1,           // [kSlots] gate producer: a (and W2) landed -> Z
    BAR_COUNT = BAR_GFULL + kSlots
};
static_assert(BAR_COUNT <= kNumBars, "barrier space");

constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColA = 0, kColP = 128, kColU = 256, kColO = 384;

enum { T_Q = 0, T_K = 1, T_V = 2, T_G = 3, kTensors = 4 };

struct TcParams {
    CUtensorMap maps[kTensors][kHeights];  // box height box_height(i)
    CUtensorMap cmaps[kTensors];           // column orders: a chunk's 64-token walk as one im2col load
    void *out;
    float *final_state;
    int H, grid_h, grid_w, order, n_chunks, T;
    int Dk, Dv;                            // multiples of 8 up to 128 (the tensors' row widths)
    int nh;                                // ceil(Dk / 64): 64-channel key halves per chunk
    int nv;                                // ceil(Dv / 64): 64-column value slices, one per CTA work unit
    int n_units;                           // work units of this launch, dealt out round-robin to the CTAs
    int seg_len;                           // chunks per segment (the last one may run past the sequence)
    int nseg;                              // segments per sequence (1: no split)
    int nsu;                               // segments per (sequence, value slice) among this launch's units
    float *summary;                        // nseg > 1: per (sequence, segment < nseg - 1) end state from zero
                                           // [Dk][Dv] and total decay [Dk], fp32
    int drop_load;                         // test hook: CTA 0 withholds its first chunk's load, so the
                                           // bounded waits run out and the call reports a timeout
    unsigned long long out_row;            // elements per token of the output, H Dv (2^31 and more at 2^24 heads)
    unsigned long long wait_limit;         // kSplitFull, one key half: the bounded waits' limit in ns
    unsigned long long *flags;             // kBalanced: per CTA, == epoch once its hand-off state (in
                                           // summary, [64][64] fp32 per CTA) is written; cleared when read
    unsigned long long epoch;              // kBalanced: nonzero, new for every launch
    FastDiv fd_per, fd_nsu, fd_H, fd_gh, fd_L;  // division by L * nh, nsu, H, grid_h, L
    FastDiv bal_n;                         // kBalanced: division by the chunks per sequence
    // gate producer (maps[T_G] then load the rank-16 projection a = x W1 instead of the gates)
    CUtensorMap w2map;                     // W2 [H][r][Dk], 16-bit, box (64 channels, r rows) SW128
    const float *gbias;                    // b [H][Dk] fp32
    float tau_inv;                         // 1 / tau
    // output gate fused into the gen warpgroups' stores (GATED): u = SiLU(r) RMSNorm(o) w
    const void *gate_r;                    // r = x W_r [B][T][H][Dv], the input dtype
    const float *gate_w;                   // RMSNorm weight [Dv]
    float gate_eps;
};

// ---------------------------------------------------------------- helpers
__device__ __forceinline__ uint32_t sw128(uint32_t row, uint32_t byte) {
    return row * 128u + ((((byte >> 4) ^ (row & 7u)) << 4) | (byte & 15u));
}
__device__ __forceinline__ uint32_t off32(uint32_t row, uint32_t col) {
    return (col >> 5) * 8192u + sw128(row, (col & 31u) * 4u);
}
// SW128 operand descriptors: K-major tiles (8-row groups 1024 B apart) and
// MN-major tiles (64-element atoms 8192 B apart).  A K step of 16 elements adds
// 32 B (2 in the address field) to a K-major descriptor and 2048 B (128) to an
// MN-major one.
__device__ __forceinline__ uint64_t kdesc(uint32_t saddr) { return smem_desc(saddr, 16, 1024, kLayoutSw128); }
__device__ __forceinline__ uint64_t mndesc(uint32_t saddr) { return smem_desc(saddr, 8192, 1024, kLayoutSw128); }
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float max_nan(float a, float b) {  // NaN when either is (fmaxf drops it)
    float y;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}
__device__ __forceinline__ float to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}
__device__ __forceinline__ uint32_t h2bits(float a, float b) {
    __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&h);
}
__device__ __forceinline__ uint32_t h2bits(f2 a) {
    const float2 x = unpack2(a);
    return h2bits(x.x, x.y);
}
__device__ __forceinline__ f2 ex2_pair(f2 a) {
    const float2 x = unpack2(a);
    return pack2(ex2(x.x), ex2(x.y));
}
__device__ __forceinline__ f2 ex2_neg_pair(f2 a) {
    const float2 x = unpack2(a);
    return pack2(ex2(-x.x), ex2(-x.y));
}

// log sigma(x) = min(x, 0) - log(1 + e), e = e^{-|x|} in (0, 1], of a pair: log(1 + e) by the hardware's
// log2 (absolute error below 2^-21 on [1, 2]), or by its series e - e^2 / 2 where e < 1e-3 (error below
// e^3 / 3), so that the relative error stays below 4e-4 before the gate is rounded to fp16.  NaN
// propagates; x = +inf gives 0, x = -inf gives -inf.  (A degree-6 polynomial for log(1 + e) / e is more
// exact and as fast, but moves the fp32 state by 2e-5.)
__device__ __forceinline__ f2 log_sigmoid_pair(f2 x) {
    const float2 v = unpack2(x);
    const float2 e = make_float2(ex2(-fabsf(v.x) * kLog2e), ex2(-fabsf(v.y) * kLog2e));
    const f2 ep = pack2(e.x, e.y), one = pack2(1.f, 1.f);
    const float2 y = unpack2(add2(one, ep));
    float l0, l1;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l0) : "f"(y.x));
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l1) : "f"(y.y));
    const float2 lg = unpack2(mul2(pack2(l0, l1), pack2(0.693147182464599609375f, 0.693147182464599609375f)));
    const float2 se = unpack2(mul2(ep, fma2(pack2(-0.5f, -0.5f), ep, one)));
    const f2 l1p = pack2(e.x < 1.0e-3f ? se.x : lg.x, e.y < 1.0e-3f ? se.y : lg.y);
    return fma2(pack2(-1.f, -1.f), l1p, pack2(fminf(v.x, 0.f), fminf(v.y, 0.f)));
}

template <typename E> struct Elem;
template <> struct Elem<__half> {
    static constexpr uint32_t fmt = kFmtF16;
    static constexpr uint16_t one = 0x3C00;
    static __device__ __forceinline__ float2 unpack(uint32_t w) {
        return __half22float2(*reinterpret_cast<const __half2 *>(&w));
    }
    static __device__ __forceinline__ uint32_t pack(float a, float b) { return h2bits(a, b); }
    static __device__ __forceinline__ f2 unpack_pair(uint32_t w) {
        const float2 x = unpack(w);
        return pack2(x.x, x.y);
    }
};
template <> struct Elem<__nv_bfloat16> {
    static constexpr uint32_t fmt = kFmtBF16;
    static constexpr uint16_t one = 0x3F80;
    static __device__ __forceinline__ float2 unpack(uint32_t w) {
        return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w));
    }
    static __device__ __forceinline__ uint32_t pack(float a, float b) {
        __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<uint32_t *>(&h);
    }
    static __device__ __forceinline__ f2 unpack_pair(uint32_t w) { return pack2(w << 16, w & 0xFFFF0000u); }
};

__device__ __forceinline__ void record_timeout(volatile uint32_t *abort_flag) {
    *abort_flag = 1u;
    atomicOr(&g_device_status, kStatusTimeout);
}

// Smem row rho of chunk c holds walk position w0 + rho, where the walk is the
// forward scan (row-major for row orders, down the columns for column orders)
// and w0 mirrors the range for reverse orders (scan position 64c + 63 - rho).
__host__ __device__ __forceinline__ int chunk_w0(int order, int T, int c) {
    return (order & 1) ? (T - kC * (c + 1)) : kC * c;
}

// Work units are (sequence, 64-column value slice) pairs.  A CTA walks the units
// blockIdx.x, blockIdx.x + gridDim.x, ... as one stream of "virtual chunks": each
// 64-token chunk of a unit appears once per 64-channel key half (Dk = 128: twice),
// carrying that half's q, k, g and the unit's v slice.  The output is linear in the
// key channels (o = sum over halves of Qtil_a S_a + P_a V), so the halves go through
// the same per-chunk pipeline and only their O products share one accumulator.
struct StreamPos {
    int bh;      // sequence b * H + h
    int vb;      // value slice
    int c;       // chunk of the sequence
    int a;       // key half
    int seg;     // segment of the sequence
    int cl;      // chunk within the segment
    bool start;  // a run of the unit starts here: its state is set
    bool hin;    // kBalanced: the run starts from the previous CTA's hand-off state
};
// Units are (sequence, segment, value slice), the value slice fastest (the two
// slices of a sequence read the same q, k and gates); a unit covers seg_len chunks.
__device__ __forceinline__ StreamPos stream_pos(int v, int L, int nh, int lognv, const FastDiv &per, bool split,
                                                const FastDiv &nsu) {
    const int j = fdiv(v, per), rem = v - j * per.d;
    const int unit = static_cast<int>(blockIdx.x) + j * static_cast<int>(gridDim.x);
    const int rest = unit >> lognv;
    const int bh = split ? fdiv(rest, nsu) : rest;
    const int seg = split ? rest - bh * nsu.d : 0;
    const int cl = rem / nh;
    const int a = rem - cl * nh;
    return {bh, unit & ((1 << lognv) - 1), seg * L + cl, a, seg, cl, cl == 0 && a == 0, false};
}

// kBalanced: the units' chunks in order, unit by unit, cut into `grid` equal contiguous
// ranges (each at least one unit long, so no range lies inside one unit), decoded once per
// CTA (`cta`; the host runs the same code for gtr_gla_balanced_walk).  A CTA first runs the head [0, c_hi) of the unit its range ends in (from zero; its
// end state goes to the next CTA), then its whole units, then the tail [c_lo, N) of the
// unit its range starts in, from the state the previous CTA handed over at the start of
// its own run (long before).
struct BalRange {
    int base_head, base_full, base_tail;  // flattened chunk index = v + the base of v's piece
    int c_hi, t0;                         // pieces: [0, c_hi) head, [c_hi, t0) whole units, [t0, G) tail
    int G;
};
__host__ __device__ __forceinline__ BalRange bal_range(int N, int n_units, int cta, int grid) {
    const long long tot = static_cast<long long>(n_units) * N;
    const long long lo = tot * cta / grid, hi = tot * (cta + 1) / grid;
    const int u_lo = static_cast<int>(lo / N), c_lo = static_cast<int>(lo - static_cast<long long>(u_lo) * N);
    const int u_hi = static_cast<int>(hi / N), c_hi = static_cast<int>(hi - static_cast<long long>(u_hi) * N);
    const int u_first = c_lo ? u_lo + 1 : u_lo;
    BalRange r;
    r.c_hi = c_hi;
    r.t0 = c_hi + (u_hi - u_first) * N;
    r.base_head = u_hi * N;                          // head: chunk v of unit u_hi
    r.base_full = u_first * N - c_hi;                // whole units from u_first on
    r.base_tail = static_cast<int>(lo) - r.t0;       // tail: chunk c_lo + (v - t0) of unit u_lo
    r.G = static_cast<int>(hi - lo);
    return r;
}
// The piece is picked by two compares and the unit by one multiply-high division; a
// three-way branch over the pieces made every role's per-chunk decode slower and cost the
// whole kernel 10 %, and an integer division here another 17 %.
__host__ __device__ __forceinline__ StreamPos stream_pos_bal(int v, int N, int lognv, int base_head, int base_full,
                                                             int base_tail, int c_hi, int t0, const FastDiv &fn) {
    const int g = v + (v < c_hi ? base_head : (v < t0 ? base_full : base_tail));
    const int unit = fdiv(g, fn), c = g - unit * N;
    const bool hin = v == t0;  // the tail's first chunk (t0 == G when there is no tail)
    return {unit >> lognv, unit & ((1 << lognv) - 1), c, 0, 0, c, c == 0 || hin, hin};
}

// kBalanced: bounded wait for the previous CTA's hand-off flag, read with acquire semantics at
// GPU scope (the writer fenced before setting it), so the waiting thread needs no fence of its
// own, which would also wait for its output stores in flight.  Out of line: it runs once per CTA.
__device__ __noinline__ bool handoff_wait(const unsigned long long *f, unsigned long long epoch,
                                          volatile uint32_t *abort_flag) {
    bool got = ld_acquire_u64(f) == epoch;
    const uint64_t t0 = global_timer_ns();
    while (!got && !*abort_flag && global_timer_ns() - t0 < kWaitLimitNs) {
        __nanosleep(64);
        got = ld_acquire_u64(f) == epoch;
    }
    return got;
}

// Visit the TMA load boxes of one chunk: calls f(map height index, smem row, c2, c3).
// Row orders: one 64-row box at token w0 (rows outside the sequence are
// zero-filled).  Column orders: boxes for each column segment, of the segment's
// exact height (at most two: its multiple of 8 and the remainder), plus zero-fill
// boxes placed past the last column for rows outside the sequence.
//
// Runs of rows down one column (at most two zero-fill runs, then the column
// segments), each loaded as at most two boxes: its multiple of 8 and the remainder.
// One call site for f keeps the producer's issue code small.
template <typename F>
__host__ __device__ __forceinline__ void chunk_load_boxes(int order, int T, const FastDiv &gh, int grid_w, int c, F &&f) {
    const int w0 = chunk_w0(order, T, c);
    if ((order >> 1) == 0) {
        f(kHeights - 1, 0, w0, 0);
        return;
    }
    if (w0 >= T || w0 + kC <= 0) {  // a padding chunk wholly past the sequence: all zeros
        f(kHeights - 1, 0, grid_w, 0);
        return;
    }
    const int lo = w0 < 0 ? 0 : w0, hi = (w0 + kC > T) ? T : w0 + kC;
    int phase = 0, w = lo;
#pragma unroll 1
    for (;;) {
        int len, row, c2, c3;
        if (phase == 0) {  // rows before the sequence: zero-fill past the last column
            phase = 1;
            if (lo <= w0) continue;
            len = lo - w0, row = 0, c2 = grid_w, c3 = 0;
        } else if (phase == 1) {  // rows after the sequence
            phase = 2;
            if (hi >= w0 + kC) continue;
            len = w0 + kC - hi, row = hi - w0, c2 = grid_w, c3 = 0;
        } else {  // the next column segment
            if (w >= hi) break;
            const int x = fdiv(w, gh), y = w - x * gh.d;
            len = gh.d - y;
            if (len > hi - w) len = hi - w;
            row = w - w0, c2 = x, c3 = y;
            w += len;
        }
        const int len8 = len & ~7;
#pragma unroll 1
        for (int part = 0; part < 2; ++part) {
            const int n = part == 0 ? len8 : len - len8;
            if (n == 0) continue;
            f(part == 0 ? 6 + n / 8 : n - 1, row + (part == 0 ? 0 : len8), c2, c3 + (part == 0 ? 0 : len8));
        }
    }
}

// Column orders, chunk c wholly inside the sequence: its 64 tokens (down column x0 from row y0
// and on into the next columns) load as one im2col walk per tensor; returns false for row orders
// and for chunks that reach past either end, which load boxes (chunk_load_boxes).
__host__ __device__ __forceinline__ bool chunk_walk_start(int order, int T, const FastDiv &gh, int c, int *x0, int *y0) {
    const int w0 = chunk_w0(order, T, c);
    if ((order >> 1) == 0 || w0 < 0 || w0 + kC > T) return false;
    *x0 = fdiv(w0, gh);
    *y0 = w0 - *x0 * gh.d;
    return true;
}

// fp16-pair mask of score columns 2e, 2e + 1 from a bit set of kept columns
__device__ __forceinline__ uint32_t pmask(uint32_t vbits, int e) {
    return (((vbits >> (2 * e)) & 1u) ? 0x0000FFFFu : 0u) | (((vbits >> (2 * e + 1)) & 1u) ? 0xFFFF0000u : 0u);
}

__device__ __forceinline__ void cp_async_16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Spatial token of walk position w (-1 outside the sequence).
__device__ __forceinline__ int walk_token(int order, int T, const FastDiv &gh, int grid_w, int w) {
    if (w < 0 || w >= T) return -1;
    if ((order >> 1) == 0) return w;
    const int x = fdiv(w, gh);
    return (w - x * gh.d) * grid_w + x;
}

// Stores a row's 32 output columns (col0 ..., four 16-byte pieces) of token t per lane, lanes l and
// l ^ 1 holding two rows.  Stored as they are, every instruction writes 16 bytes into each of 32
// sectors; the pair first swaps pieces so that its two lanes write 32 consecutive bytes of one row
// (GB300, graph replays: 6,400 tokens 170 -> 155 us, 704^2 images with Dk = 32 42 -> 39 us, B = 32,
// H = 12, 40 x 40 87 -> 84 us; a 4 x 4 transpose to 64 bytes costs more instructions than it gives).
// With two key halves and split sequences the epi has no registers left for it (252 us against 255 at
// 128 x 128; whole sequences 198 -> 185 us).
template <typename E, bool PAIR>
__device__ __forceinline__ void store_row(const TcParams &p, const uint32_t (&ow)[16], int b, int h, int t, int col0) {
    if constexpr (PAIR) {
        uint4 pc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) pc[q] = make_uint4(ow[4 * q], ow[4 * q + 1], ow[4 * q + 2], ow[4 * q + 3]);
        const bool odd = threadIdx.x & 1;
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
            // the even lane gives its odd pieces for the odd lane's even ones
            uint4 s = odd ? pc[q] : pc[q + 1];
            s.x = __shfl_xor_sync(0xffffffffu, s.x, 1);
            s.y = __shfl_xor_sync(0xffffffffu, s.y, 1);
            s.z = __shfl_xor_sync(0xffffffffu, s.z, 1);
            s.w = __shfl_xor_sync(0xffffffffu, s.w, 1);
            if (odd) pc[q] = s;
            else pc[q + 1] = s;
        }
        // now pc[q] is the even lane's row and pc[q + 1] the odd lane's, at piece q + odd
        const int other = __shfl_xor_sync(0xffffffffu, t, 1);
        const int t0 = odd ? other : t, t1 = odd ? t : other;
        const int col = col0 + 8 * odd;
        const size_t ld = p.out_row;
        E *base = static_cast<E *>(p.out) + ((size_t)b * p.T * p.H + h) * p.Dv + col;
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
            if (col + 8 * q < p.Dv) {  // (columns past Dv and rows outside the sequence stay behind)
                if (t0 >= 0) *reinterpret_cast<uint4 *>(base + t0 * ld + 8 * q) = pc[q];
                if (t1 >= 0) *reinterpret_cast<uint4 *>(base + t1 * ld + 8 * q) = pc[q + 1];
            }
        }
    } else if (t >= 0) {
        uint4 *dst = reinterpret_cast<uint4 *>(static_cast<E *>(p.out) + (((size_t)b * p.T + t) * p.H + h) * p.Dv + col0);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (col0 + 8 * q < p.Dv) dst[q] = make_uint4(ow[4 * q], ow[4 * q + 1], ow[4 * q + 2], ow[4 * q + 3]);
    }
}

// Exact scores for one chunk (extreme or non-finite log-decays) by CUDA cores, for any decay: serial
// prefix a of the clamped gates (log2), then P[rho][sigma] = sum_i q k 2^{a_r,i - a_j,i} (j <= r)
// without a split that could overflow.  For a key block J of 16 scan positions before the row's own,
// 2^{a_r - a_j} = 2^{a_r - a_e} 2^{a_e - a_j} with e the block's last position: both factors are at most
// 1, the second one is formed once per key (kb), the first for every eight keys of a row.  The row's own block
// does the same with blocks of 4, and only keys in the row's own 4 take an exponential each: about 670
// per row instead of 2,080 on average (128 for kb, 192 and 96 for the row's factors in earlier blocks of 16
// and 4, 256 in its own 4; a block of 16 is done in two halves, each with the row's factors anew) (GB300, 6,400 tokens with the gate producer and strong decays
// 2,065 -> 1,367 us; B = 4, H = 8, 48 x 40, all chunks exact, 265 -> 170 us).  Also Qtil = q 2^{a},
// Kbar = k 2^{a_last - a}, and the chunk decay.  `as` holds two 64 x 64 fp32 arrays, a and kb, whose
// rows' float4s are permuted so that a warp's 16 rows fall into different banks.  SUM (summary passes): no scores and no queries, the q and gate tiles stay as they are.
__device__ __forceinline__ float4 &exact_at(float *base, int row, int i) {  // channels i .. i + 3 (i % 4 == 0)
    return *reinterpret_cast<float4 *>(base + row * kD + (((i >> 2) ^ (row & 15)) << 2));
}
template <typename E, typename GT, bool SUM>
__device__ __noinline__ void exact_chunk(uint8_t *tq, uint8_t *tk, uint8_t *tgate, float *as,
                                         float *decay, int rev, int tg, int bar_id) {
    float *kb = as + kC * kD;
    if (tg < kD) {
        float run = 0.f;
#pragma unroll 4
        for (int r = 0; r < kC; ++r) {
            const int rho = rev ? kC - 1 - r : r;
            const uint16_t bits = *reinterpret_cast<const uint16_t *>(tgate + sw128(rho, tg * 2));
            float x = Elem<GT>::unpack(bits).x * kLog2e;
            x = x < kGateMinLog2 ? kGateMinLog2 : x;
            run += x;
            (&exact_at(as, rho, tg & ~3).x)[tg & 3] = run;
        }
        decay[tg] = ex2(run);
    }
    named_barrier_sync(bar_id, 128);
    const int rho = tg >> 1, half = tg & 1;
    const int r = rev ? kC - 1 - rho : rho;
    uint32_t packed[16];  // the row's 32 scores of this half, pairs in shared-memory order
    if constexpr (!SUM) {
        auto row_at = [&](int pos) { return rev ? kC - 1 - pos : pos; };  // tile row of a scan position
        auto pair16 = [&](const uint8_t *tile, int row, int i) {
            return Elem<E>::unpack(*reinterpret_cast<const uint32_t *>(tile + sw128(row, i * 2)));
        };
        // kb = k 2^{a_e - a}, e the last position of the key's block of `n`
        auto make_kb = [&](int n) {
            const int re = row_at(r | (n - 1));
#pragma unroll 1
            for (int i = half * 32; i < half * 32 + 32; i += 4) {
                const float4 a = exact_at(as, rho, i), ae = exact_at(as, re, i);
                const float2 k0 = pair16(tk, rho, i), k1 = pair16(tk, rho, i + 2);
                exact_at(kb, rho, i) = make_float4(k0.x * ex2(ae.x - a.x), k0.y * ex2(ae.y - a.y),
                                                   k1.x * ex2(ae.z - a.z), k1.y * ex2(ae.w - a.w));
            }
        };
        // acc[c] += sum_i q_i 2^{a_r,i - a_e,i} kb[j0 + c][i] over channels [i0, i1), c < N, for the keys of
        // a block that ends at position epos
        auto dense = [&](auto &acc, int i0, int i1, int j0, int epos) {
            constexpr int N = sizeof(acc) / sizeof(float);
            const int re = row_at(epos);
#pragma unroll 1
            for (int i = i0; i < i1; i += 4) {
                const float4 a = exact_at(as, rho, i), ae = exact_at(as, re, i);
                const float2 q0 = pair16(tq, rho, i), q1 = pair16(tq, rho, i + 2);
                const f2 w0 = pack2(q0.x * ex2(a.x - ae.x), q0.y * ex2(a.y - ae.y));
                const f2 w1 = pack2(q1.x * ex2(a.z - ae.z), q1.y * ex2(a.w - ae.w));
#pragma unroll
                for (int c = 0; c < N; ++c) {
                    const float4 k = exact_at(kb, row_at(j0 + c), i);
                    const float2 t = unpack2(fma2(w0, pack2(k.x, k.y), mul2(w1, pack2(k.z, k.w))));
                    acc[c] += t.x + t.y;
                }
            }
        };
        make_kb(16);
        named_barrier_sync(bar_id, 128);
        const int I = r >> 4;  // the row's block (the same for a warp's 16 rows)
#pragma unroll 1
        for (int b4 = 0; b4 < 4; ++b4) {  // eight columns of a block at a time (few registers: the callers keep theirs)
            const int sb = 2 * half + (b4 >> 1), J = rev ? 3 - sb : sb, j0 = 16 * J + 8 * (rev ? 1 - (b4 & 1) : (b4 & 1));
            float acc[8] = {};
            if (J < I) dense(acc, 0, kD, j0, 16 * J + 15);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                packed[4 * b4 + e] = rev ? h2bits(acc[7 - 2 * e], acc[6 - 2 * e]) : h2bits(acc[2 * e], acc[2 * e + 1]);
        }
        named_barrier_sync(bar_id, 128);  // every use of kb is done
        make_kb(4);
        named_barrier_sync(bar_id, 128);
        // the row's own block: each of the row's two threads takes half of the channels
        const int sbI = rev ? 3 - I : I;
#pragma unroll 1
        for (int J4 = 0; J4 < 4; ++J4) {
            float acc[4] = {};
            const int j0 = 16 * I + 4 * J4;
            if (j0 < (r & ~3)) {
                dense(acc, 32 * half, 32 * half + 32, j0, j0 + 3);
            }
            if (j0 == (r & ~3)) {  // the row's own four: an exponential per channel
#pragma unroll 1
                for (int i = 32 * half; i < 32 * half + 32; i += 4) {
                    const float4 a = exact_at(as, rho, i);
                    const float2 q0 = pair16(tq, rho, i), q1 = pair16(tq, rho, i + 2);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int rj = row_at(j0 + c);
                        const float4 aj = exact_at(as, rj, i);
                        const float2 k0 = pair16(tk, rj, i), k1 = pair16(tk, rj, i + 2);
                        const float t = q0.x * k0.x * ex2(a.x - aj.x) + q0.y * k0.y * ex2(a.y - aj.y) +
                                        q1.x * k1.x * ex2(a.z - aj.z) + q1.y * k1.y * ex2(a.w - aj.w);
                        if (j0 + c <= r) acc[c] += t;  // (later keys' exponents are positive)
                    }
                }
            }
            __syncwarp();
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], 1);
            if (sbI >> 1 == half) {  // columns 4 J4 .. of the block, in shared-memory order
                uint32_t *dst = packed + 8 * (sbI & 1) + (rev ? 2 * (3 - J4) : 2 * J4);
                dst[0] = rev ? h2bits(acc[3], acc[2]) : h2bits(acc[0], acc[1]);
                dst[1] = rev ? h2bits(acc[1], acc[0]) : h2bits(acc[2], acc[3]);
            }
        }
    }
    const int rho_last = rev ? 0 : kC - 1;
    named_barrier_sync(bar_id, 128);  // every q/k/gate read of this chunk is done
    if constexpr (!SUM) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            *reinterpret_cast<uint4 *>(tgate + sw128(rho, (half * 32 + 8 * q) * 2)) =
                make_uint4(packed[4 * q], packed[4 * q + 1], packed[4 * q + 2], packed[4 * q + 3]);
    }
#pragma unroll 1
    for (int i = half * 32; i < half * 32 + 32; i += 4) {
        const float4 a = exact_at(as, rho, i), l = exact_at(as, rho_last, i);
        uint2 *kp = reinterpret_cast<uint2 *>(tk + sw128(rho, i * 2));
        const uint2 kw = *kp;
        const float2 k0 = Elem<E>::unpack(kw.x), k1 = Elem<E>::unpack(kw.y);
        if constexpr (!SUM) {
            uint2 *qp = reinterpret_cast<uint2 *>(tq + sw128(rho, i * 2));
            const uint2 qw = *qp;
            const float2 q0 = Elem<E>::unpack(qw.x), q1 = Elem<E>::unpack(qw.y);
            *qp = make_uint2(h2bits(q0.x * ex2(a.x), q0.y * ex2(a.y)), h2bits(q1.x * ex2(a.z), q1.y * ex2(a.w)));
        }
        *kp = make_uint2(h2bits(k0.x * ex2(l.x - a.x), k0.y * ex2(l.y - a.y)),
                         h2bits(k1.x * ex2(l.z - a.z), k1.y * ex2(l.w - a.w)));
    }
}

// Operands of a tf32-mode chunk (split factors beyond the fp16 range): tf32 Q^ and
// K^ for the score product in the group's operand buffer, fp16 Qtil = Q^ c1 over q and
// Kbar = K^ c2 over k.  Re-reads the thread's log-decays from TMEM (A is kept until the operands are
// built), half of them at a time in a loop: this rarer path is out of line, and what it costs the
// chunks that take it is its code and the registers its callers lose (GB300, 6,400 tokens: all 32
// log-decays at once 163 us fp16 and 172 us bf16, two halves in a loop with packed pairs 150 and 159;
// inlined it cost B = 32, H = 12, 40 x 40 6 %).
// SUM (summary passes): only Kbar.
template <typename E, bool SUM>
__device__ __noinline__ void tf32_operands(uint8_t *tq, uint8_t *tk, uint8_t *opbuf, const float *ref,
                                           uint32_t taddr, int row, int ch0) {
    uint8_t *qh = opbuf, *kh = opbuf + kTile32;
#pragma unroll 1
    for (int hf = 0; hf < 2; ++hf) {
        uint32_t ar[16];
        tmem_ld_16x32bx2_x16(taddr + 16 * hf, ar);
        tmem_ld_wait();
#pragma unroll
        for (int g8 = 0; g8 < 2; ++g8) {
            const int cl = ch0 + 16 * hf + 8 * g8;
            const uint32_t o16 = sw128(row, cl * 2);
            const uint4 qw = SUM ? make_uint4(0u, 0u, 0u, 0u) : *reinterpret_cast<const uint4 *>(tq + o16);
            const uint4 kw = *reinterpret_cast<const uint4 *>(tk + o16);
            const uint32_t qa[4] = {qw.x, qw.y, qw.z, qw.w}, ka[4] = {kw.x, kw.y, kw.z, kw.w};
            // A_mid, c1 and c2 of the 8 channels (16-byte aligned rows of the references)
            f2 am[4], c1v[4], c2v[4];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(ref + cl + 4 * e);
                const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(ref + 2 * kD + cl + 4 * e);
                const ulonglong2 c = *reinterpret_cast<const ulonglong2 *>(ref + 3 * kD + cl + 4 * e);
                am[2 * e] = a.x, am[2 * e + 1] = a.y;
                c1v[2 * e] = b.x, c1v[2 * e + 1] = b.y;
                c2v[2 * e] = c.x, c2v[2 * e + 1] = c.y;
            }
            f2 q2[4], k2[4];
            float qs[8], ks[8];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const f2 x = fma2(pack2(ar[8 * g8 + 2 * e], ar[8 * g8 + 2 * e + 1]), pack2(kLog2e, kLog2e),
                                  mul2(am[e], pack2(-kLog2e, -kLog2e)));
                q2[e] = mul2(Elem<E>::unpack_pair(qa[e]), ex2_pair(x));
                k2[e] = mul2(Elem<E>::unpack_pair(ka[e]), ex2_neg_pair(x));
                const float2 a = unpack2(q2[e]), b = unpack2(k2[e]);
                qs[2 * e] = a.x, qs[2 * e + 1] = a.y;
                ks[2 * e] = b.x, ks[2 * e + 1] = b.y;
            }
            if (!SUM) {
                *reinterpret_cast<float4 *>(qh + off32(row, cl)) =
                    make_float4(to_tf32(qs[0]), to_tf32(qs[1]), to_tf32(qs[2]), to_tf32(qs[3]));
                *reinterpret_cast<float4 *>(qh + off32(row, cl + 4)) =
                    make_float4(to_tf32(qs[4]), to_tf32(qs[5]), to_tf32(qs[6]), to_tf32(qs[7]));
                *reinterpret_cast<float4 *>(kh + off32(row, cl)) =
                    make_float4(to_tf32(ks[0]), to_tf32(ks[1]), to_tf32(ks[2]), to_tf32(ks[3]));
                *reinterpret_cast<float4 *>(kh + off32(row, cl + 4)) =
                    make_float4(to_tf32(ks[4]), to_tf32(ks[5]), to_tf32(ks[6]), to_tf32(ks[7]));
            }
            uint32_t qo[4], ko[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                qo[e] = h2bits(mul2(q2[e], c1v[e]));
                ko[e] = h2bits(mul2(k2[e], c2v[e]));
            }
            if (!SUM) *reinterpret_cast<uint4 *>(tq + o16) = make_uint4(qo[0], qo[1], qo[2], qo[3]);
            *reinterpret_cast<uint4 *>(tk + o16) = make_uint4(ko[0], ko[1], ko[2], ko[3]);
        }
    }
}

// GP (gate producer, one key half, whole sequences): the gates are not read but computed
// from the rank-16 projection, g = logsigmoid(a W2 + b) / tau (Sec. 3.1, retention gate):
// Z = a W2 by one MMA into the chunk's TMEM A buffer, g by the gen warpgroup that owns the
// chunk, written as fp16 over the chunk's gate tile, then A = L G as usual (fp16).
// GATED (outputs stored by the gen warpgroups, one key half, one value slice): the stores
// apply the output gate u = SiLU(r) * RMSNorm(o) * w of Sec. 3.1 to the row's fp32 outputs
// (the deployed kernel's fused epilogue, App. C.3), so o is rounded once, as u.
template <typename E, int NH, int NV, int MODE, bool GENOUT, bool GP = false, bool GATED = false>
__global__ void __launch_bounds__(kThreads, 1) gla_tc_kernel(const __grid_constant__ TcParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                ~static_cast<uintptr_t>(1023));
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kOffBar);
    volatile uint32_t *tmem_base_s = reinterpret_cast<volatile uint32_t *>(smem + kOffMisc);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(smem + kOffMisc + 4);
    float *decay_s = reinterpret_cast<float *>(smem + kOffDecay);
    volatile uint32_t *mode_s = reinterpret_cast<volatile uint32_t *>(smem + kOffMode);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Two key halves: the epi holds two states and spills at the 128 registers a thread of 512 gets, so
    // the roles are aligned to warpgroups (0-3 producer and issuers, 4-11 gen, 12-15 epi) and the
    // control warps' registers go to the others (GB300, Dk = Dv = 128: 128 x 128 images 219 -> 202 us,
    // B = 16, H = 12, 40 x 40 185 -> 163 us).  With one key half nothing spills, and the roles as listed
    // at the top measured faster (6,400 tokens, tf32 scores: 159 us against 164 aligned).
    constexpr bool kAligned = NH == 2;
    constexpr int kGen0 = kAligned ? 4 : 2, kEpi0 = kAligned ? 12 : 10, kWarpPU = kAligned ? 2 : 14;
    constexpr uint32_t kRegsCtl = 64, kRegsGen = 136, kRegsEpi = 176;
    static_assert(kRegsCtl + 2 * kRegsGen + kRegsEpi == 4 * 128, "the registers of the launch");
    // the output pass after a summary pass may start now: its CTAs set up (barriers, TMEM) on
    // the free SMs and wait for this grid only before they read the summaries
    if constexpr (MODE == kSummary) pdl_launch_dependents();
    // MODE kFull / kSplitFull: outputs (a split sequence's later segments start from
    // the state folded from the segment summaries).  MODE kSummary: per segment only
    // the end state from zero and the total decay (k, v and gates; no scores or outputs).
    constexpr bool kSum = MODE == kSummary;
    constexpr bool kSplit = MODE == kSplitFull || MODE == kSummary;
    constexpr bool kBal = MODE == kBalanced;
    static_assert(!kBal || NH == 1, "balanced ranges hand over one key half's state");
    static_assert(!GP || (NH == 1 && MODE == kFull), "the gate producer runs whole sequences, one key half");
    static_assert(!GATED || (GENOUT && NH == 1 && NV == 1 && MODE != kSummary), "the fused gate normalises whole rows");
    // element type of the gate tile: the loaded gates, or the fp16 gates the gate producer writes
    using GE = typename std::conditional<GP, __half, E>::type;
    // GENOUT (one key half, outputs): the gen warpgroup that built a chunk also reads its
    // outputs back from TMEM and stores them, while it waits for the P of its next chunk,
    // which takes that work off the epi's serial per-chunk chain.  The host selects it where
    // that was measured faster (fp16 launches of at most one wave); elsewhere the epi stores.
    constexpr bool kGenOut = GENOUT && NH == 1 && !kSum;
    // The SM's instruction cache is shared by all roles (ncu: 4 % of its requests miss on B = 32, H = 12,
    // 40 x 40 and at Dk = Dv = 128, 14 % with the gate producer).  The fp16 operand build therefore runs as a loop over two halves of a thread's channels, each read from TMEM when
    // its turn comes, where the epi stores the outputs (GB300, graph replays: 84.5 -> 82.3 us there,
    // Dk = Dv = 128 188 -> 185 us); unrolled it is faster where the gen warps store them (6,400 tokens,
    // tf32 scores: 155 us against 171).
    constexpr bool kRollBuild = !kGenOut;
    const int N = p.n_chunks;   // chunks per sequence
    const int L = p.seg_len;    // chunks per unit
    // Summaries of two key halves: a unit is one half with every value slice (else one value slice
    // with every key half), so that a chunk's A and Kbar are built once instead of once per slice.  The
    // second slice of v takes the q tile's place, its U the O columns (neither is used by a summary),
    // its state the other half's registers.  GB300, Dk = Dv = 128, 128 x 128, B = 2, H = 8: 252 -> 219 us both passes.
    constexpr bool kHalfSum = kSum && NH == 2;
    constexpr int kSlices = kHalfSum ? NV : 1;  // value slices per virtual chunk
    constexpr int nh = kHalfSum ? 1 : NH;   // 64-channel key halves per chunk (Dk / 64) of a unit
    constexpr int lognv = kHalfSum ? 1 : NV - 1;  // units per (sequence, segment): 64-column value slices, or key halves
    constexpr int kDk = 64 * NH, kDv = 64 * NV;
    // this CTA's stream of virtual chunks: every barrier phase, stage slot and TMEM
    // buffer below follows the stream index (O: the real chunk's index), so
    // consecutive units flow through one pipeline
    BalRange br{};
    if constexpr (kBal) br = bal_range(N, p.n_units, static_cast<int>(blockIdx.x), static_cast<int>(gridDim.x));
    const int b_head = br.base_head, b_full = br.base_full, b_tail = br.base_tail, b_chi = br.c_hi, b_t0 = br.t0;
    const int G = kBal ? br.G
                       : L * nh *
                             ((p.n_units - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) /
                              static_cast<int>(gridDim.x));
    auto pos = [&](int v) -> StreamPos {
        if constexpr (kBal) return stream_pos_bal(v, N, lognv, b_head, b_full, b_tail, b_chi, b_t0, p.bal_n);
        StreamPos ps = stream_pos(v, L, nh, lognv, p.fd_per, kSplit, p.fd_nsu);
        if constexpr (kHalfSum) {
            ps.a = ps.vb;
            ps.vb = 0;
        }
        return ps;
    };
    const int rev = p.order & 1;
    // kSplitFull, one key half: the CTA may start long before the summary pass ends, and in segments past
    // the first its roles' waits depend on the start state the epi folds from the summaries (from the third
    // chunk on; the readout: from the first).  So their limit is the launch's: 1 s and the time that pass
    // may take at most.  (Waiting for the grid in every role, or a limit that starts when the epi has seen
    // it end, cost 0.1 to 0.5 us of an 11 us call and 2 % of 80 us ones.)
    const uint64_t limit = MODE == kSplitFull && NH == 1 ? p.wait_limit : kWaitLimitNs;

    if (threadIdx.x == 0) {
        *abort_flag = 0u;
        for (int i = 0; i < kSlots; ++i) {
            mbar_init(&bars[BAR_FULL + i], 1);
            mbar_init(&bars[BAR_GFULL + i], 1);
            mbar_init(&bars[BAR_EMPTY + i], MODE == kSummary ? 1 : 2);  // after U(c) and after O(c)
            mbar_init(&bars[BAR_REFS + i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars[BAR_AFULL + i], 1);
            mbar_init(&bars[BAR_PURDY + i], 8);
            mbar_init(&bars[BAR_PFULL + i], 1);
            mbar_init(&bars[BAR_UFULL + i], 1);
            mbar_init(&bars[BAR_ORDY + i], 8);
            mbar_init(&bars[BAR_OFULL + i], 1);
            mbar_init(&bars[BAR_ZFULL + i], 1);
            mbar_init(&bars[BAR_GRDY + i], 4);
        }
        mbar_init(&bars[BAR_SIN], 4);
        mbar_init(&bars[BAR_DONE], 3);  // one commit per issuer warp
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(const_cast<uint32_t *>(tmem_base_s), kTmemCols);
        tmem_relinquish();
    }
    if (warp >= kGen0 && warp < kGen0 + 4) {
        // triangle of ones in scan order: L[rho][sigma] = 1 when sigma is at or before rho
        const int tg = threadIdx.x - 32 * kGen0;
        const int rho = tg >> 1, half = tg & 1;
        uint8_t *L = smem + kOffL;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int s0 = half * 32 + u * 8 + 2 * e;
                const bool k0 = rev ? (s0 >= rho) : (s0 <= rho);
                const bool k1 = rev ? (s0 + 1 >= rho) : (s0 + 1 <= rho);
                w[e] = (k0 ? (uint32_t)Elem<GE>::one : 0u) | ((k1 ? (uint32_t)Elem<GE>::one : 0u) << 16);
            }
            *reinterpret_cast<uint4 *>(L + sw128(rho, (half * 32 + u * 8) * 2)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        fence_proxy_async_smem();
    }
    // kSplitFull, two key halves (one: see the epi): the start state of the CTA's segment (a split
    // launch gives every CTA one segment), folded from the summaries of the segments before it by all 512 threads, each
    // taking 8 of a key half's 64 x 64 values and walking the summaries from the latest back
    // (S_start = sum_s' (prod_{s' < s'' < seg} Diag(D_s'')) S_end(s'), Eq. chunk_boundary_main
    // across segments) with several summaries' loads in flight.  A serial fold by the epi alone
    // waited one L2 round trip per summary, about 8 us for the 13th segment.  The result lands in
    // gen warpgroup 0's tf32 operand buffer, which the epi reads on entry; the group writes the
    // buffer only after the epi's arrival on named barrier kBarSin.
    if constexpr (MODE == kSplitFull && NH == 2) {
        pdl_wait();  // the summaries are the previous grid's: this launch may start before it ends
        const StreamPos p0 = pos(0);
        if (G > 0 && p0.seg > 0) {
            float *sin = reinterpret_cast<float *>(smem + kOffOp);  // [NH][64 rows][64 columns] fp32
            const size_t stride = (size_t)kDk * kDv + kDk;
            const float *base = p.summary + (size_t)p0.bh * (p.nseg - 1) * stride;
            const int r = threadIdx.x >> 3, col = (threadIdx.x & 7) * 8;
#pragma unroll
            for (int a = 0; a < NH; ++a) {
                float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                float coef = 1.f;
#pragma unroll 4
                for (int s2 = p0.seg - 1; s2 >= 0; --s2) {
                    const float *bs = base + (size_t)s2 * stride;
                    const float4 *x = reinterpret_cast<const float4 *>(bs + (size_t)(64 * a + r) * kDv + 64 * p0.vb + col);
                    const float4 x0 = x[0], x1 = x[1];
                    const float d = bs[(size_t)kDk * kDv + 64 * a + r];
                    acc[0] = fmaf(coef, x0.x, acc[0]);
                    acc[1] = fmaf(coef, x0.y, acc[1]);
                    acc[2] = fmaf(coef, x0.z, acc[2]);
                    acc[3] = fmaf(coef, x0.w, acc[3]);
                    acc[4] = fmaf(coef, x1.x, acc[4]);
                    acc[5] = fmaf(coef, x1.y, acc[5]);
                    acc[6] = fmaf(coef, x1.z, acc[6]);
                    acc[7] = fmaf(coef, x1.w, acc[7]);
                    coef *= d;
                }
                float4 *dst = reinterpret_cast<float4 *>(sin + (64 * a + r) * 64 + col);
                dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
                dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
            }
        }
    }
    tc_fence_before();
    // Warp 0, which initialised the mbarriers, goes on to load the first chunks while the others wait
    // for each other's set-up (0.5 us of a launch; GB300, graph replays: B = 1, H = 6, 40 x 40 fp16
    // 13.8 -> 13.5 us, B = 4, H = 12 bf16 28.2 -> 27.4, B = 32 80.5 -> 80.0)
    if (warp == 0)
        named_barrier_arrive(kBarSetup, kThreads);
    else
        named_barrier_sync(kBarSetup, kThreads);
    tc_fence_after();
    const uint32_t tmem = *tmem_base_s;  // (warp 0 does not use it)

    if (kAligned ? warp < 4 : (warp < 2 || warp >= 14)) {
        if constexpr (kAligned) setmaxnreg_dec<kRegsCtl>();
        if (warp == 0) {
            // ======================================================= TMA producer
            if (lane == 0) {
                int issued = 0;
                for (int g = 0; g < G; ++g) {
                    const int sl = g % kSlots;
                    const StreamPos ps = pos(g);
                    const int b = fdiv(ps.bh, p.fd_H), h = ps.bh - b * p.H, c = ps.c;
                    const int xk = 64 * ps.a, xv = 64 * ps.vb;  // channel offsets of the key half, value slice
                    if (!mbar_wait(&bars[BAR_EMPTY + sl], ((g / kSlots) & 1) ^ 1, abort_flag, limit)) {
                        record_timeout(abort_flag);
                        break;
                    }
                    // (slots 2 and 3 serve the start state's fold first)
                    if (MODE == kSplitFull && NH == 1 && g == 2 && ps.seg > 0 && !mbar_wait(&bars[BAR_SIN], 0, abort_flag, limit)) {
                        record_timeout(abort_flag);
                        break;
                    }
                    uint8_t *st = smem + kOffSlot + sl * kSlotBytes;
                    uint64_t *fb = &bars[BAR_FULL + sl];
                    if (!(p.drop_load && blockIdx.x == 0 && g == 0)) {
                        // gate producer: a unit's first chunk also brings the head's W2 block, into the
                        // buffer of the unit's parity (the unit before last, whose Z products used it,
                        // ended at least four chunks earlier: its last Z completed before this slot freed)
                        const bool w2 = GP && ps.cl == 0;
                        // (the a tile and W2 go first and have their own mbarrier: Z and the gates need nothing
                        // else; B = 32, H = 12, 40 x 40 bf16 125.5 -> 122.5 us.  The same for loaded gates: 2 to
                        // 3 % slower at B = 8, H = 16, 80 x 80 and at Dk = Dv = 128, 1 % faster at B = 32)
                        uint64_t *gb = GP ? &bars[BAR_GFULL + sl] : fb;
                        if (GP) mbar_arrive_expect_tx(gb, kTile16 + (w2 ? kW2Bytes : 0));
                        mbar_arrive_expect_tx(fb, GP || (kSum && kSlices == 1) ? kSlotBytes - kTile16 : kSlotBytes);
                        if (w2) tma_load_5d(smem + kOffW2 + (fdiv(g, p.fd_L) & 1) * kW2Bytes, &p.w2map, gb, 0, 0, h, 0, 0);
                        int x0, y0;
                        if (chunk_walk_start(p.order, p.T, p.fd_gh, c, &x0, &y0)) {
                            // column orders, chunk inside the sequence: one im2col walk per tensor
                            // (boxes per column segment cost the TMA unit one request each and ran
                            // up to 1.9x slower)
                            if (GP) tma_load_im2col_5d(st + kG, &p.cmaps[T_G], gb, 0, y0, x0, 0, b);
                            if (!kSum) tma_load_im2col_5d(st + kQ, &p.cmaps[T_Q], fb, xk, y0, x0, h, b);
                            tma_load_im2col_5d(st + kK, &p.cmaps[T_K], fb, xk, y0, x0, h, b);
                            tma_load_im2col_5d(st + kV, &p.cmaps[T_V], fb, xv, y0, x0, h, b);
                            if (kSlices == 2) tma_load_im2col_5d(st + kQ, &p.cmaps[T_V], fb, 64, y0, x0, h, b);
                            if (!GP) tma_load_im2col_5d(st + kG, &p.cmaps[T_G], fb, xk, y0, x0, h, b);
                        } else chunk_load_boxes(p.order, p.T, p.fd_gh, p.grid_w, c, [&](int hi, int row, int c2, int c3) {
                            // gate producer: the 16 projection values of each token, zero-filled to a 128-byte row
                            if (GP) tma_load_5d(st + kG + row * 128, &p.maps[T_G][hi], gb, 0, 0, c2, c3, b);
                            if (!kSum) tma_load_5d(st + kQ + row * 128, &p.maps[T_Q][hi], fb, xk, h, c2, c3, b);
                            tma_load_5d(st + kK + row * 128, &p.maps[T_K][hi], fb, xk, h, c2, c3, b);
                            tma_load_5d(st + kV + row * 128, &p.maps[T_V][hi], fb, xv, h, c2, c3, b);
                            if (kSlices == 2) tma_load_5d(st + kQ + row * 128, &p.maps[T_V][hi], fb, 64, h, c2, c3, b);
                            if (!GP) tma_load_5d(st + kG + row * 128, &p.maps[T_G][hi], fb, xk, h, c2, c3, b);
                        });
                    }
                    ++issued;
                }
                if (*abort_flag) {  // never leave while copies are still landing in shared memory
                    for (int g = (issued > kSlots ? issued - kSlots : 0); g < issued; ++g)
                        if (!(p.drop_load && blockIdx.x == 0 && g == 0)) {
                            mbar_wait(&bars[BAR_FULL + g % kSlots], (g / kSlots) & 1, nullptr, kWaitLimitNs);
                            if (GP) mbar_wait(&bars[BAR_GFULL + g % kSlots], (g / kSlots) & 1, nullptr, kWaitLimitNs);
                        }
                }
            }
        } else {
            // ======================================================= MMA issuers
            // Three warps issue the products, each in program order and waiting only for
            // its own inputs, so that the issue overhead of one product never delays
            // another.  A whole warp runs each loop (operands warp-uniform) and one
            // elected lane issues each MMA.
            //   warp 1   A(c) = L G          once chunk c landed and gen(c-2) built its
            //                                operands (so TMEM A of the parity was read)
            //   warp 14  P(c) = Q^ K^^T,     once PURDY(c): gen(c) operands in smem and epi
            //            U(c) = Kbar^T V     drained U(c-2)
            //   warp 15  O(c) = Q S'_[c] + P V   once ORDY(c)
            // A tcgen05.commit tracks only its own thread's MMAs: the slot of chunk c is
            // released by two commits, after U(c) (warp 14) and after O(c) (warp 15); P(c)
            // and A(c) completed before ORDY(c).  No waiter can be overtaken by two phases
            // of its barrier: PURDY(c + 2) needs A(c + 2) and U(c), FULL of the next chunk
            // of a slot needs that slot's EMPTY, ORDY(c + 2) needs O(c) read.
            const uint32_t slot0 = smem_u32(smem + kOffSlot);
            bool ok = true;
            if (warp == 1) {
                const uint32_t idesc_a = instr_desc(Elem<GE>::fmt, 64, 64, 0, 1);
                const uint64_t dL = kdesc(smem_u32(smem + kOffL));

                for (int c = 0; c < G; ++c) {
                    if constexpr (GP) {
                        // the gen group wrote the chunk's gates (over its a tile, whose Z it has read)
                        ok = !__any_sync(0xffffffffu, !mbar_wait(&bars[BAR_GRDY + (c & 1)], (c >> 1) & 1, abort_flag, limit));
                        if (!ok) break;
                    } else {
                        if (c >= 2) {
                            ok = !__any_sync(0xffffffffu, !mbar_wait(&bars[BAR_PURDY + (c & 1)], ((c - 2) >> 1) & 1, abort_flag, limit));
                            if (!ok) break;
                        }
                        ok = !__any_sync(0xffffffffu, !mbar_wait(&bars[BAR_FULL + c % kSlots], (c / kSlots) & 1, abort_flag, limit));
                        if (!ok) break;
                    }
                    tc_fence_after();
                    const uint64_t dg = mndesc(slot0 + (c % kSlots) * kSlotBytes + kG);
                    mma4_f16_ss_warp<2, 128>(tmem + kColA + (c & 1) * 64, dL, dg, idesc_a, 0);
                    mma_commit_warp(&bars[BAR_AFULL + (c & 1)]);
                }
            } else if (warp == kWarpPU) {
                const uint32_t idesc_p16 = instr_desc(kFmtF16, 64, 64, 0, 0);
                const uint32_t idesc_p32 = instr_desc(kFmtTF32, 64, 64, 0, 0);
                const uint32_t idesc_u = instr_desc(kFmtF16, 64, 64, 1, 1);
                const uint64_t dqh0 = kdesc(smem_u32(smem + kOffOp)), dkh0 = kdesc(smem_u32(smem + kOffOp + kTile32));
                int su = 0;
                // GP: Z(c) = a W2 (M = 64 tokens, N = 64 channels, K = r = 16: one MMA) into chunk c's TMEM A
                // buffer; a tile K-major with 128-byte rows, W2 MN-major
                auto issue_z = [&](int c) {
                    const uint64_t da = kdesc(slot0 + (c % kSlots) * kSlotBytes + kG);
                    const uint64_t dw = mndesc(smem_u32(smem + kOffW2) + (fdiv(c, p.fd_L) & 1) * kW2Bytes);
                    mma_f16_ss_warp(tmem + kColA + (c & 1) * 64, da, dw, instr_desc(Elem<E>::fmt, 64, 64, 0, 1), 0);
                    mma_commit_warp(&bars[BAR_ZFULL + (c & 1)]);
                };
                auto full = [&](int c) -> uint64_t * { return &bars[BAR_GFULL + c % kSlots]; };
                if constexpr (GP) {
                    for (int c = 0; c < 2 && c < G; ++c) {
                        ok = !__any_sync(0xffffffffu, !mbar_wait(full(c), 0, abort_flag, limit));
                        if (!ok) break;
                        tc_fence_after();
                        issue_z(c);
                    }
                }
                for (int c = 0; ok && c < G; ++c) {
                    ok = !__any_sync(0xffffffffu, !mbar_wait(&bars[BAR_PURDY + (c & 1)], (c >> 1) & 1, abort_flag, limit));
                    if (!ok) break;
                    tc_fence_after();
                    // GP: chunk c + 2's Z reuses the A buffer that gen(c) has read.  It goes before P(c) and
                    // U(c) when the chunk has landed (the gen group forms those gates while it waits for P(c)),
                    // else after them.
                    bool z_due = GP && c + 2 < G;
                    if (z_due && !__any_sync(0xffffffffu, !mbar_test(full(c + 2), ((c + 2) / kSlots) & 1))) {
                        issue_z(c + 2);
                        z_due = false;
                    }
                    const uint32_t st = slot0 + su * kSlotBytes;
                    const uint32_t mode = __shfl_sync(0xffffffffu, mode_s[su], 0);
                    const uint32_t dp = tmem + kColP + (c & 1) * 64;
                    if (kSum) {
                        // summaries need no scores
                    } else if (mode == kModeF16) {
                        const uint64_t dq = kdesc(st + kQ), dk = kdesc(st + kK);
                        mma4_f16_ss_warp<2, 2>(dp, dq, dk, idesc_p16, 0);
                        mma_commit_warp(&bars[BAR_PFULL + (c & 1)]);
                    } else if (mode == kModeTF32) {
                        const uint64_t dqh = dqh0 + (c & 1) * (2 * kTile32 >> 4), dkh = dkh0 + (c & 1) * (2 * kTile32 >> 4);
                        mma4_tf32_ss_warp(dp, dqh, dkh, idesc_p32, 0);
                        mma4_tf32_ss_warp(dp, dqh + 512, dkh + 512, idesc_p32, 1);  // (the second 32 columns: 8192 B >> 4)
                        mma_commit_warp(&bars[BAR_PFULL + (c & 1)]);
                    } else if (lane == 0) {
                        mbar_arrive(&bars[BAR_PFULL + (c & 1)]);  // exact scores are already in smem
                    }
                    __syncwarp();
                    // U(c) = Kbar^T V (fp16 mode: K^^T V): the k tile read as the MN-major A
                    const uint64_t dk = mndesc(st + kK), dv = mndesc(st + kV);
                    const uint32_t du = tmem + kColU + (c & 1) * 64;
                    mma4_f16_ss_warp<128, 128>(du, dk, dv, idesc_u, 0);
                    if (kSlices == 2) mma4_f16_ss_warp<128, 128>(tmem + kColO + (c & 1) * 64, dk, mndesc(st + kQ), idesc_u, 0);
                    mma_commit2_warp(&bars[BAR_UFULL + (c & 1)], &bars[BAR_EMPTY + su]);  // U is the slot's last reader among this warp's MMAs
                    su = (su == kSlots - 1) ? 0 : su + 1;
                    if (z_due) {
                        ok = !__any_sync(0xffffffffu, !mbar_wait(full(c + 2), ((c + 2) / kSlots) & 1, abort_flag, limit));
                        if (!ok) break;
                        tc_fence_after();
                        issue_z(c + 2);
                    }
                }
            } else if (!kSum) {
                const uint32_t idesc_o = instr_desc(kFmtF16, 64, 64, 0, 1);
                const uint32_t sbuf = smem_u32(smem + kOffS);
                int so = 0;
                for (int c = 0; c < G; ++c) {
                    ok = !__any_sync(0xffffffffu, !mbar_wait(&bars[BAR_ORDY + (c & 1)], (c >> 1) & 1, abort_flag, limit));
                    if (!ok) break;
                    tc_fence_after();
                    // O(c) = Qtil S_[c] + P V  (fp16 mode: Q^ (Diag(c1) S_[c]) + P V); the key
                    // halves of one real chunk accumulate into the same TMEM buffer
                    const uint32_t st = slot0 + so * kSlotBytes;
                    const uint64_t dq = kdesc(st + kQ), ds = mndesc(sbuf + (c & 1) * kTile16);
                    const uint64_t dpm = kdesc(st + kG), dv = mndesc(st + kV);
                    const uint32_t d = tmem + kColO + ((c / nh) & 1) * 64;
                    const uint32_t acc0 = (c % nh) != 0;
                    mma4_f16_ss_warp<2, 128>(d, dq, ds, idesc_o, acc0);
                    mma4_f16_ss_warp<2, 128>(d, dpm, dv, idesc_o, 1);
                    mma_commit2_warp(&bars[BAR_OFULL + (c & 1)], &bars[BAR_EMPTY + so]);  // every product of the slot's chunk is done
                    so = (so == kSlots - 1) ? 0 : so + 1;
                }
            }
            if (!ok && lane == 0) record_timeout(abort_flag);
            mma_commit_warp(&bars[BAR_DONE]);  // TMEM is released only after every MMA completed
            mbar_wait(&bars[BAR_DONE], 0, nullptr, kWaitLimitNs);
        }
    } else if (warp < kEpi0) {
        if constexpr (kAligned) setmaxnreg_inc<kRegsGen>();
        // ======================================================= gen warpgroups (chunks c = gw mod 2)
        const int gw = (warp - kGen0) >> 2;      // 0: even chunks, 1: odd chunks
        const int bar_id = 1 + gw;
        if constexpr (MODE == kSplitFull && NH == 2) {
            if (gw == 0) named_barrier_sync(kBarSin, 256);  // the epi took the folded start state
        }
        const int q4 = warp & 3, hc = lane >> 4;
        const int row = 16 * q4 + (lane & 15);   // smem row rho of this thread's accumulator row
        const int ch0 = 32 * hc;                 // its 32 key channels (A) / score columns (P)
        const uint32_t lane_base = static_cast<uint32_t>(32 * q4) << 16;
        const int tg = threadIdx.x - 32 * kGen0 - 128 * gw;
        const int rho_mid = rev ? 32 : 31, rho_last = rev ? 0 : 63;
        // causal mask of this thread's 32 score columns as packed fp16-pair masks (scan order)
        uint32_t vbits = 0u;  // bit s: score column ch0 + s is kept
        for (int s = 0; s < 32; ++s)
            if (rev ? (ch0 + s >= row) : (ch0 + s <= row)) vbits |= 1u << s;
        // outputs of chunk co (this group's) once O(co) completed: TMEM -> this thread's row at its
        // token's spatial position; false when the wait gave up
        auto gen_out = [&](int co) {
            // (a lane whose wait gave up goes on with the others, as what follows is warp-collective; the group
            // leaves together at the barrier of its next chunk, and the outputs are then undefined)
            if (!mbar_wait(&bars[BAR_OFULL + (co & 1)], (co >> 1) & 1, abort_flag, limit)) record_timeout(abort_flag);
            tc_fence_after();
            uint32_t r[32];
            tmem_ld_16x32bx2_x16(tmem + lane_base + kColO + (co & 1) * 64 + 0, *reinterpret_cast<uint32_t(*)[16]>(&r[0]));
            tmem_ld_16x32bx2_x16(tmem + lane_base + kColO + (co & 1) * 64 + 16, *reinterpret_cast<uint32_t(*)[16]>(&r[16]));
            tmem_ld_wait();
            uint32_t ow[16];
            const StreamPos po = pos(co);
            const int b = fdiv(po.bh, p.fd_H), h = po.bh - b * p.H;
            const int t = walk_token(p.order, p.T, p.fd_gh, p.grid_w, chunk_w0(p.order, p.T, po.c) + row);
            if constexpr (GATED) {
                // u = SiLU(r) * o / sqrt(mean_j o_j^2 + eps) * w over the head's Dv outputs: this
                // thread holds 32 of the row's columns, the lane 16 apart the other 32 (padded
                // columns are 0 and count for nothing)
                uint4 rq[4] = {};
                const E *rrow = static_cast<const E *>(p.gate_r) + (((size_t)b * p.T + (t < 0 ? 0 : t)) * p.H + h) * p.Dv;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (t >= 0 && ch0 + 8 * q < p.Dv) rq[q] = *reinterpret_cast<const uint4 *>(rrow + ch0 + 8 * q);
                float ss = 0.f;
#pragma unroll
                for (int j = 0; j < 32; ++j) ss = fmaf(__uint_as_float(r[j]), __uint_as_float(r[j]), ss);
                ss += __shfl_xor_sync(0xffffffffu, ss, 16);
                const float inv = rsqrtf(ss / static_cast<float>(p.Dv) + p.gate_eps);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float wq[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                    if (ch0 + 8 * q < p.Dv) {
                        *reinterpret_cast<float4 *>(&wq[0]) = __ldg(reinterpret_cast<const float4 *>(p.gate_w + ch0 + 8 * q));
                        *reinterpret_cast<float4 *>(&wq[4]) = __ldg(reinterpret_cast<const float4 *>(p.gate_w + ch0 + 8 * q + 4));
                    }
                    const uint32_t rw[4] = {rq[q].x, rq[q].y, rq[q].z, rq[q].w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 z = Elem<E>::unpack(rw[e]);
                        const float s0 = __fdividef(z.x, 1.f + __expf(-z.x)), s1 = __fdividef(z.y, 1.f + __expf(-z.y));
                        const float o0 = __uint_as_float(r[8 * q + 2 * e]), o1 = __uint_as_float(r[8 * q + 2 * e + 1]);
                        ow[4 * q + e] = Elem<E>::pack(s0 * o0 * inv * wq[2 * e], s1 * o1 * inv * wq[2 * e + 1]);
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) ow[j] = Elem<E>::pack(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
            }
            store_row<E, true>(p, ow, b, h, t, 64 * po.vb + ch0);
        };
        // GP: chunk cz's gates from Z = a W2 (Sec. 3.1): g = logsigmoid(z + b) / tau in fp32, written as
        // fp16 over the a tile, whose Z product has completed; rows outside the sequence keep g = 0 (no
        // decay), as zero-filled gate rows do.  Done while the group waits for its previous chunk's
        // scores, so that A = L G is ready when that chunk is finished (before, its round trip and the
        // gates stood at the start of every chunk: GB300, B = 32, H = 12, 40 x 40 bf16 182 -> 127 us).
        auto make_gates = [&](int cz) {
            const int zb = cz & 1;
            // the position and the bias of the thread's channels first: their loads land while Z does
            // (loaded where they are added, B = 32 127.6 us against 125.9, B = 1, H = 6 fp16 42.4 against 40.4)
            const StreamPos pz = pos(cz);
            const int wz = chunk_w0(p.order, p.T, pz.c) + row;
            const uint32_t live = wz >= 0 && wz < p.T ? 0xffffffffu : 0u;
            const float *bz = p.gbias + (size_t)(pz.bh - fdiv(pz.bh, p.fd_H) * p.H) * p.Dk + ch0;
            ulonglong2 bq[8];  // (Dk is a multiple of 8: a block of 8 channels is all inside it or all past it)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                bq[2 * q] = bq[2 * q + 1] = make_ulonglong2(0ull, 0ull);
                if (ch0 + 8 * q < p.Dk) {
                    bq[2 * q] = __ldg(reinterpret_cast<const ulonglong2 *>(bz + 8 * q));
                    bq[2 * q + 1] = __ldg(reinterpret_cast<const ulonglong2 *>(bz + 8 * q + 4));
                }
            }
            // (a lane whose wait gave up goes on with the others, as the TMEM loads are warp-collective; the
            // group leaves together at the barrier of its next chunk)
            if (!mbar_wait(&bars[BAR_ZFULL + zb], (cz >> 1) & 1, abort_flag, limit)) record_timeout(abort_flag);
            tc_fence_after();
            uint8_t *gt = smem + kOffSlot + (cz % kSlots) * kSlotBytes + kG;
            uint32_t zr[32];
            tmem_ld_16x32bx2_x16(tmem + lane_base + kColA + zb * 64 + 0, *reinterpret_cast<uint32_t(*)[16]>(&zr[0]));
            tmem_ld_16x32bx2_x16(tmem + lane_base + kColA + zb * 64 + 16, *reinterpret_cast<uint32_t(*)[16]>(&zr[16]));
            tmem_ld_wait();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const f2 bb[4] = {bq[2 * q].x, bq[2 * q].y, bq[2 * q + 1].x, bq[2 * q + 1].y};
                uint32_t gq[4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    gq[e] = h2bits(mul2(log_sigmoid_pair(add2(pack2(zr[8 * q + 2 * e], zr[8 * q + 2 * e + 1]), bb[e])),
                                        pack2(p.tau_inv, p.tau_inv))) & live;
                *reinterpret_cast<uint4 *>(gt + sw128(row, (ch0 + 8 * q) * 2)) = make_uint4(gq[0], gq[1], gq[2], gq[3]);
            }
            fence_proxy_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars[BAR_GRDY + zb]);  // this warp's rows of G are in smem
        };
        if constexpr (GP) {
            if (gw < G) make_gates(gw);
        }
        int last_c = -1;  // the group's last chunk completed (its outputs are stored after the loop)
        for (int c = gw; c < G; c += 2) {
            const int sl = c % kSlots, bb = c & 1;
            const uint32_t ph = (c >> 1) & 1;
            uint8_t *st = smem + kOffSlot + sl * kSlotBytes;
            bool fail = !mbar_wait(&bars[BAR_AFULL + bb], ph, abort_flag, limit);
            // (gate producer: A(c) waited for the a tile only)
            if constexpr (GP) fail = fail || !mbar_wait(&bars[BAR_FULL + sl], (c / kSlots) & 1, abort_flag, limit);
            // bf16 values become fp16 MMA operands in place (exact for |v| in the fp16
            // normal range); the loads go first so that their latency hides behind the
            // operand build, the converted words are stored with the operands
            tc_fence_after();
            const uint32_t ta = tmem + lane_base + kColA + bb * 64;
            // references of chunk c: [0,64) raw A_mid, [64,128) raw A_last, [128,192) c1 = 2^{A_mid},
            // [192,256) c2 = 2^{A_last - A_mid}
            float *ref = reinterpret_cast<float *>(smem + kOffRef) + sl * kRefFloats;
            auto write_refs = [&](const uint32_t (&a)[32]) {
                if (!fail && (row == rho_mid || row == rho_last)) {
                    float *dst = ref + (row == rho_mid ? 0 : kD) + ch0;
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        reinterpret_cast<float4 *>(dst)[q] = make_float4(__uint_as_float(a[4 * q]), __uint_as_float(a[4 * q + 1]),
                                                                         __uint_as_float(a[4 * q + 2]), __uint_as_float(a[4 * q + 3]));
                }
            };
            uint32_t ar[32];  // the thread's log-decays (unused with kRollBuild)
            if constexpr (kRollBuild) {
                if (q4 == rho_mid >> 4 || q4 == rho_last >> 4) {  // (the warps of the reference rows)
                    uint32_t a[32];
                    tmem_ld_16x32bx2_x16(ta + 0, *reinterpret_cast<uint32_t(*)[16]>(&a[0]));
                    tmem_ld_16x32bx2_x16(ta + 16, *reinterpret_cast<uint32_t(*)[16]>(&a[16]));
                    tmem_ld_wait();
                    write_refs(a);
                }
            } else {
                tmem_ld_16x32bx2_x16(ta + 0, *reinterpret_cast<uint32_t(*)[16]>(&ar[0]));
                tmem_ld_16x32bx2_x16(ta + 16, *reinterpret_cast<uint32_t(*)[16]>(&ar[16]));
                tmem_ld_wait();
                write_refs(ar);
            }
            tc_fence_before();
            if (named_barrier_or(bar_id, 128, fail || *abort_flag != 0u)) {  // the group gives up together
                record_timeout(abort_flag);
                break;
            }
            // every warp reduces the split range M over the 64 channels itself (no second
            // barrier); warp 0 of the group writes the constants the readout and epi use
            uint32_t mode;
            {
                const float am0 = ref[lane] * kLog2e, al0 = ref[kD + lane] * kLog2e;
                const float am1 = ref[lane + 32] * kLog2e, al1 = ref[kD + lane + 32] * kLog2e;
                // a gate of -inf after the middle leaves A_mid = NaN (0 x -inf in A = L G) and A_last = -inf:
                // both terms of its channel are NaN, which must not get lost in the maximum
                float m = max_nan(max_nan(-am0, am0 - al0), max_nan(-am1, am1 - al1));
                if (!(m <= 3.0e38f)) m = 3.0e38f;  // NaN / inf gates: exact path
                // (m >= 0 for log gates <= 0, so its bits order like the values.)  One redux instead of five
                // shuffles and maxima: every warp waits for this, 1.13x at Dk = Dv = 128 and 1.04x at
                // B = 32, H = 12, 40 x 40 on a GB300
                m = __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(m)));
                mode = m <= kMaxRefF16 ? kModeF16 : (m <= kMaxRefTF32 ? kModeTF32 : kModeExact);
                if (tg < 32) {
                    ref[2 * kD + lane] = ex2(am0);
                    ref[2 * kD + lane + 32] = ex2(am1);
                    ref[3 * kD + lane] = ex2(al0 - am0);
                    ref[3 * kD + lane + 32] = ex2(al1 - am1);
                    decay_s[sl * kD + lane] = ex2(al0);
                    decay_s[sl * kD + lane + 32] = ex2(al1);
                    if (tg == 0) mode_s[sl] = mode;
                    __syncwarp();
                    // constants and mode of chunk c -> epi, written by this warp
                    if (tg == 0 && mode != kModeExact) mbar_arrive(&bars[BAR_REFS + sl]);
                }
            }
            uint8_t *tq = st + kQ, *tk = st + kK, *tgt = st + kG;
            bool opfail = false;
            if (mode != kModeF16) {
                // the constants written by warp 0 above are read by every warp of the group; the
                // group's own operand buffer was last read by P(c - 2), complete before mask(c - 2)
                opfail = named_barrier_or(bar_id, 128, false);
            }
            if (mode == kModeF16) {
                // the operands of channels cl .. cl + 7, whose log-decays are a[i0 ...]
                auto build8 = [&](const auto &a, int i0, int cl) {
                    const ulonglong2 am0 = *reinterpret_cast<const ulonglong2 *>(ref + cl);  // raw A_mid of 8 channels
                    const ulonglong2 am1 = *reinterpret_cast<const ulonglong2 *>(ref + cl + 4);
                    const f2 am[4] = {am0.x, am0.y, am1.x, am1.y};
                    // packed pairs of channels: the same roundings in two thirds of the instructions (GB300,
                    // graph replays, with the epi's state packed too: B = 32, H = 12, 40 x 40 1.03x in
                    // bf16 and 1.07x in fp16, Dk = Dv = 128 1.13x)
                    const uint32_t o16 = sw128(row, cl * 2);
                    const uint4 qw = kSum ? make_uint4(0u, 0u, 0u, 0u) : *reinterpret_cast<const uint4 *>(tq + o16);
                    const uint4 kw = *reinterpret_cast<const uint4 *>(tk + o16);
                    const uint32_t qa[4] = {qw.x, qw.y, qw.z, qw.w}, ka[4] = {kw.x, kw.y, kw.z, kw.w};
                    uint32_t qo[4], ko[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const f2 x = fma2(pack2(a[i0 + 2 * e], a[i0 + 2 * e + 1]), pack2(kLog2e, kLog2e),
                                          mul2(am[e], pack2(-kLog2e, -kLog2e)));
                        qo[e] = h2bits(mul2(Elem<E>::unpack_pair(qa[e]), ex2_pair(x)));
                        ko[e] = h2bits(mul2(Elem<E>::unpack_pair(ka[e]), ex2_neg_pair(x)));
                    }
                    // Q^ over q, K^ over k (each thread rewrites exactly what it read)
                    if (!kSum) *reinterpret_cast<uint4 *>(tq + o16) = make_uint4(qo[0], qo[1], qo[2], qo[3]);
                    *reinterpret_cast<uint4 *>(tk + o16) = make_uint4(ko[0], ko[1], ko[2], ko[3]);
                };
                if constexpr (kRollBuild) {
#pragma unroll 1
                    for (int hf = 0; hf < 2; ++hf) {
                        uint32_t a[16];
                        tmem_ld_16x32bx2_x16(ta + 16 * hf, a);
                        tmem_ld_wait();
#pragma unroll
                        for (int g8 = 0; g8 < 2; ++g8) build8(a, 8 * g8, ch0 + 16 * hf + 8 * g8);
                    }
                } else {
#pragma unroll
                    for (int g8 = 0; g8 < 4; ++g8) build8(ar, 8 * g8, ch0 + 8 * g8);
                }
            } else if (!opfail) {
                if (mode == kModeTF32)
                    tf32_operands<E, kSum>(tq, tk, smem + kOffOp + gw * 2 * kTile32, ref, ta, row, ch0);
                else
                    exact_chunk<E, GE, kSum>(tq, tk, tgt, reinterpret_cast<float *>(smem + kOffOp + gw * 2 * kTile32), decay_s + sl * kD, rev, tg,
                                   bar_id);
            }
            if constexpr (std::is_same<E, __nv_bfloat16>::value) {
#pragma unroll 1
                for (int vs = 0; vs < kSlices; ++vs) {
                    uint8_t *tv = vs == 0 ? st + kV : st + kQ;
                    uint4 vw[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) vw[q] = *reinterpret_cast<const uint4 *>(tv + sw128(row, (ch0 + 8 * q) * 2));
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t *wp = reinterpret_cast<uint32_t *>(&vw[q]);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float2 fv = Elem<E>::unpack(wp[e]);
                            wp[e] = h2bits(fv.x, fv.y);
                        }
                        *reinterpret_cast<uint4 *>(tv + sw128(row, (ch0 + 8 * q) * 2)) = vw[q];
                    }
                }
            }
            fence_proxy_async_smem();
            tc_fence_before();
            // (no group barrier: every thread rewrote only what it read, and each warp signals its own rows;
            // an exact chunk's decays are the whole group's)
            if (mode == kModeExact) {
                if (named_barrier_or(bar_id, 128, opfail)) {
                    record_timeout(abort_flag);
                    break;
                }
                if (tg == 0) mbar_arrive(&bars[BAR_REFS + sl]);  // constants and mode of chunk c -> epi
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars[BAR_PURDY + bb]);  // operands in smem, A(c) read
            if (kSum) continue;  // no scores
            if constexpr (GP) {
                if (c + 2 < G) make_gates(c + 2);
            }
            // ---- outputs of the group's previous chunk c-2 (O(c) reuses its TMEM buffer only
            // after ORDY(c), which this group signals below)
            if constexpr (kGenOut) {
                if (c >= 2) gen_out(c - 2);
            }
            // ---- masked scores of chunk c over its gate tile (consumed by A(c) long ago)
            // (a warp that gives up here skips the rest of the chunk; the group leaves together at
            // the barrier of its next one)
            const bool pfail = !mbar_wait(&bars[BAR_PFULL + bb], ph, abort_flag, limit);
            if (__any_sync(0xffffffffu, pfail)) {
                if (lane == 0) record_timeout(abort_flag);
                continue;
            }
            if (mode != kModeExact) {
                tc_fence_after();
                uint32_t r[32];
                tmem_ld_16x32bx2_x16(tmem + lane_base + kColP + bb * 64 + 0, *reinterpret_cast<uint32_t(*)[16]>(&r[0]));
                tmem_ld_16x32bx2_x16(tmem + lane_base + kColP + bb * 64 + 16, *reinterpret_cast<uint32_t(*)[16]>(&r[16]));
                tmem_ld_wait();
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    *reinterpret_cast<uint4 *>(tgt + sw128(row, (ch0 + 8 * q) * 2)) = make_uint4(
                        h2bits(__uint_as_float(r[8 * q + 0]), __uint_as_float(r[8 * q + 1])) & pmask(vbits, 4 * q + 0),
                        h2bits(__uint_as_float(r[8 * q + 2]), __uint_as_float(r[8 * q + 3])) & pmask(vbits, 4 * q + 1),
                        h2bits(__uint_as_float(r[8 * q + 4]), __uint_as_float(r[8 * q + 5])) & pmask(vbits, 4 * q + 2),
                        h2bits(__uint_as_float(r[8 * q + 6]), __uint_as_float(r[8 * q + 7])) & pmask(vbits, 4 * q + 3));
            }
            tc_fence_before();
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars[BAR_ORDY + bb]);  // this warp's rows of P are in smem
            last_c = c;
        }
        if constexpr (kGenOut) {
            if (last_c >= 0 && last_c + 2 >= G) gen_out(last_c);
        }
    } else {
        // ======================================================= epi warpgroup (warps 10-13)
        if constexpr (kAligned) setmaxnreg_inc<kRegsEpi>();
        // Carries the fp32 state of the current key half in registers (thread: channel
        // row, 32 value columns; with two key halves the other half's state waits in So
        // and the two swap after every virtual chunk), writes Diag(c1) S for the readout
        // product, folds U into the state, and stores each real chunk's outputs at its
        // tokens' spatial positions once the O product of its last key half completed.
        const int q4 = warp & 3, hc = lane >> 4;
        const int row = 16 * q4 + (lane & 15);   // channel i for U / S, token rho for O
        const int ch0 = 32 * hc;
        const uint32_t lane_base = static_cast<uint32_t>(32 * q4) << 16;
        f2 S[16], So[NH == 2 ? 16 : 1];  // packed pairs of columns
#pragma unroll
        for (int j = 0; j < 16; ++j) S[j] = 0ull;
        if constexpr (NH == 2) {
#pragma unroll
            for (int j = 0; j < 16; ++j) So[j] = 0ull;
        }
        if constexpr (MODE == kSplitFull && NH == 2) {  // the start state the whole CTA folded (segments past the first)
            if (G > 0 && pos(0).seg > 0) {
                const f2 *sin = reinterpret_cast<const f2 *>(smem + kOffOp) + (row * 64 + ch0) / 2;
#pragma unroll
                for (int j = 0; j < 16; ++j) S[j] = sin[j];
#pragma unroll
                for (int j = 0; j < 16; ++j) So[j] = sin[64 * 32 + j];
            }
            named_barrier_arrive(kBarSin, 256);  // gen warpgroup 0 may now use its operand buffer
        }
        float dp = 1.f, dpo = 1.f;  // summaries: the segment's decay product per key half
        const size_t sum_stride = (size_t)kDk * kDv + kDk;
        bool ok = true;
        if (lane == 0) {  // TMEM U buffers start out free: the drains of chunks -2 and -1
            mbar_arrive(&bars[BAR_PURDY + 0]);
            mbar_arrive(&bars[BAR_PURDY + 1]);
        }
        // kSplitFull, one key half: the start state of the CTA's segment (a split launch gives every CTA
        // one segment), folded from the summaries of the segments before it, from the latest back
        // (S_start = sum_s' (prod_{s' < s'' < seg} Diag(D_s'')) S_end(s'), Eq. chunk_boundary_main across
        // segments), while the first two chunks load and go through the gen warps: only their S' needs it.
        // Bound by the L2 reads (16 KB a summary, 64 B a cycle into the SM): cp.async keeps four summaries
        // in flight, in the slots of chunks 2 and 3, which the producer leaves alone until BAR_SIN.  Each
        // thread takes the float4s te + 128 j of a summary (rows of whole sectors) and reads back only its
        // own copies; the products of decays, one row a thread, go through the S' buffers.  GB300, graph
        // replays, against a fold by all 512 threads before the first chunk: fp16 B = 1, H = 6, 40 x 40 (13
        // segments) 13.5 -> 11.2 us, with the gate 14.7 -> 12.9; 20 x 20 12.8 -> 10.4; bf16 44 x 44 17.1 ->
        // 16.4; B = 4, H = 12, 40 x 40 (3 segments of 9 chunks) the same 27.5.
        if constexpr (MODE == kSplitFull && NH == 1) {
            const int seg = pos(0).seg;
            if (seg > 0) {
                const StreamPos p0 = pos(0);
                pdl_wait();  // the summaries are the previous grid's: this launch may start before it ends
                const int te = threadIdx.x - 32 * kEpi0;
                const int fr = te >> 4, fc = (te & 15) * 4;
                float *ring = reinterpret_cast<float *>(smem + kOffSlot + 2 * kSlotBytes);  // 4 x [64][64]
                float *coefs = reinterpret_cast<float *>(smem + kOffS);                     // [kFoldBatch][64]
                const float *last = p.summary + ((size_t)p0.bh * (p.nseg - 1) + seg - 1) * sum_stride;
                const float *src = last + (size_t)fr * kDv + 64 * p0.vb + fc, *dec = last + (size_t)kDk * kDv + te;
                auto fetch = [&](int i) {  // the i-th summary from the latest (one group each, empty past the first)
                    if (i < seg) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            cp_async_16(ring + (i & 3) * 4096 + (j * 128 + te) * 4, src - i * sum_stride + (size_t)8 * j * kDv);
                    }
                    cp_async_commit();
                };
#pragma unroll 1
                for (int i = 0; i < 4; ++i) fetch(i);
                float4 acc[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                float run = 1.f;  // te < 64: row te's product of the decays so far
                for (int i0 = 0; i0 < seg; i0 += kFoldBatch) {
                    const int m = seg - i0 < kFoldBatch ? seg - i0 : kFoldBatch;
                    if (te < 64) {
                        for (int i1 = 0; i1 < m; i1 += 8) {
                            float d[8];
#pragma unroll
                            for (int k = 0; k < 8; ++k) d[k] = i1 + k < m ? __ldcg(dec - (i0 + i1 + k) * sum_stride) : 1.f;
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                coefs[(i1 + k) * 64 + te] = run;
                                run *= d[k];
                            }
                        }
                    }
                    named_barrier_sync(3, 128);
#pragma unroll 1
                    for (int i = 0; i < m; ++i) {
                        cp_async_wait<3>();
                        const float *st = ring + ((i0 + i) & 3) * 4096 + te * 4;
                        const float *cf = coefs + i * 64 + fr;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float4 x = *reinterpret_cast<const float4 *>(st + j * 512);
                            const float cj = cf[8 * j];
                            acc[j].x = fmaf(cj, x.x, acc[j].x);
                            acc[j].y = fmaf(cj, x.y, acc[j].y);
                            acc[j].z = fmaf(cj, x.z, acc[j].z);
                            acc[j].w = fmaf(cj, x.w, acc[j].w);
                        }
                        fetch(i0 + i + 4);
                    }
                    named_barrier_sync(3, 128);  // the coefficients and (last batch) the ring are free
                }
                // to the layout of S, through the ring (rows 272 bytes apart: no bank conflicts)
#pragma unroll
                for (int j = 0; j < 8; ++j) *reinterpret_cast<float4 *>(ring + (fr + 8 * j) * kFoldPitch + fc) = acc[j];
                named_barrier_sync(3, 128);
                const ulonglong2 *sin = reinterpret_cast<const ulonglong2 *>(ring + row * kFoldPitch + ch0);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const ulonglong2 w = sin[j];
                    S[2 * j] = w.x;
                    S[2 * j + 1] = w.y;
                }
                fence_proxy_async_smem();  // the ring's slots are TMA destinations next
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[BAR_SIN]);
            }
        }
        // kBalanced: the loop runs in three pieces (head run, whole units, tail run) with the
        // hand-offs between them, so that the per-chunk loop itself carries no hand-off code
        // (in the loop it slowed every chunk: the SM's instruction cache is shared by all roles)
        const int cut0 = kBal ? b_chi : G + 1, cut1 = kBal ? b_t0 : G + 1;
        int c = 0;
        StreamPos cur{};  // chunk c's position (one decode a chunk: the outputs' is the iteration's before)
        // Every epi warp passes the pieces' boundaries, also one that gave up (its warps decide on
        // their own inside the loop): the hand-offs' named barriers then always see all four.
#pragma unroll 1
        for (int piece = 0; piece < (kBal ? 3 : 1); ++piece) {
            if (kBal && piece == 2 && b_t0 < G) {
                // the tail run starts from the previous CTA's hand-off: one thread waits for its
                // flag (bounded) and clears it for the next launch; the barrier orders the other
                // threads' reads after its acquire
                unsigned long long *f = p.flags + blockIdx.x - 1;
                bool got = true;
                if (ok && threadIdx.x == kEpi0 * 32) {
                    got = handoff_wait(f, p.epoch, abort_flag);
                    if (got) *reinterpret_cast<volatile unsigned long long *>(f) = 0ull;
                }
                if (named_barrier_or(3, 128, !ok || !got)) ok = false;  // the epi gives up together
            }
            if (kBal && piece == 2 && b_t0 < G && ok) {
                const float4 *x = reinterpret_cast<const float4 *>(p.summary + (size_t)(blockIdx.x - 1) * kD * kD +
                                                                   (size_t)row * kD + ch0);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4 w = __ldcg(x + j);  // from L2: another SM wrote it
                    S[2 * j] = pack2(w.x, w.y);
                    S[2 * j + 1] = pack2(w.z, w.w);
                }
            }
            const int c_end = piece == 0 ? cut0 : (piece == 1 ? cut1 : G + 1);
            for (; ok && c < c_end; ++c) {
                const StreamPos po = cur;  // chunk c - 1
                if (c < G) {
                    const int sl = c % kSlots, bb = c & 1;
                    const uint32_t ph = (c >> 1) & 1;
                    const StreamPos ps = cur = pos(c);
                    if (ps.start) {  // a run of a unit starts: its state (every key half)
                        if (kBal && ps.hin) {
                            // S holds the previous CTA's hand-off (taken before this piece)
                        } else if (!kSplit || kSum || ps.seg == 0) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) S[j] = 0ull;
                            if constexpr (NH == 2) {
#pragma unroll
                                for (int j = 0; j < 16; ++j) So[j] = 0ull;
                            }
                        }  // (else: a split launch gives every CTA one segment, and S holds the fold)
                        dp = dpo = 1.f;
                    }
                    bool fail = !mbar_wait(&bars[BAR_REFS + sl], (c / kSlots) & 1, abort_flag, limit);
                    // buffer bb was last read by O(c-2) (epi outputs with one key half: observed by
                    // the readout of the previous iteration already)
                    if (!kSum && (NH == 2 || kGenOut) && c >= 2)
                        fail = fail || !mbar_wait(&bars[BAR_OFULL + bb], ph ^ 1, abort_flag, limit);
                    if (__any_sync(0xffffffffu, fail)) {  // the warp leaves together
                        ok = false;
                        break;
                    }
                    const float *ref = reinterpret_cast<const float *>(smem + kOffRef) + sl * kRefFloats;
                    const bool fold = (mode_s[sl] == kModeF16);
                    const float c1 = fold ? ref[2 * kD + row] : 1.f;
                    const float c2 = fold ? ref[3 * kD + row] : 1.f;
                    const float dc = decay_s[sl * kD + row];
                    if (!kSum) {
                        // S'_[c] = Diag(c1) S_[c] (fp16, MN-major B of the readout)
                        uint8_t *sb = smem + kOffS + bb * kTile16;
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            *reinterpret_cast<uint4 *>(sb + sw128(row, (ch0 + 8 * q) * 2)) =
                                make_uint4(h2bits(mul2(S[4 * q], pack2(c1, c1))), h2bits(mul2(S[4 * q + 1], pack2(c1, c1))),
                                           h2bits(mul2(S[4 * q + 2], pack2(c1, c1))), h2bits(mul2(S[4 * q + 3], pack2(c1, c1))));
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&bars[BAR_ORDY + bb]);  // with the outputs of c-2 read out
                    }
                    // state carry: S_[c+1] = Diag(d_c) S_[c] + Diag(c2) U_c
                    fail = !mbar_wait(&bars[BAR_UFULL + bb], ph, abort_flag, limit);
                    if (__any_sync(0xffffffffu, fail)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    if constexpr (NH == 2) {  // two states live: read U in halves to save registers
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            uint32_t r[16];
                            if constexpr (kSlices == 2) {
                                tmem_ld_16x32bx2_x16(tmem + lane_base + kColO + bb * 64 + 16 * hf, r);
                                tmem_ld_wait();
#pragma unroll
                                for (int j = 0; j < 8; ++j)
                                    So[8 * hf + j] = fma2(pack2(dc, dc), So[8 * hf + j], mul2(pack2(c2, c2), pack2(r[2 * j], r[2 * j + 1])));
                            }
                            tmem_ld_16x32bx2_x16(tmem + lane_base + kColU + bb * 64 + 16 * hf, r);
                            tmem_ld_wait();
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                S[8 * hf + j] = fma2(pack2(dc, dc), S[8 * hf + j], mul2(pack2(c2, c2), pack2(r[2 * j], r[2 * j + 1])));
                        }
                    } else {
                        uint32_t r[32];
                        tmem_ld_16x32bx2_x16(tmem + lane_base + kColU + bb * 64 + 0, *reinterpret_cast<uint32_t(*)[16]>(&r[0]));
                        tmem_ld_16x32bx2_x16(tmem + lane_base + kColU + bb * 64 + 16, *reinterpret_cast<uint32_t(*)[16]>(&r[16]));
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 16; ++j) S[j] = fma2(pack2(dc, dc), S[j], mul2(pack2(c2, c2), pack2(r[2 * j], r[2 * j + 1])));
                    }
                    tc_fence_before();
                    if (kSum) {
                        dp *= dc;
                        if (ps.cl == L - 1) {  // the segment's summary
                            float *base = p.summary + ((size_t)ps.bh * (p.nseg - 1) + ps.seg) * sum_stride;
                            ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(base + (size_t)(64 * ps.a + row) * kDv + 64 * ps.vb + ch0);
#pragma unroll
                            for (int j = 0; j < 8; ++j) dst[j] = make_ulonglong2(S[2 * j], S[2 * j + 1]);
                            if constexpr (kSlices == 2) {
#pragma unroll
                                for (int j = 0; j < 8; ++j) dst[16 + j] = make_ulonglong2(So[2 * j], So[2 * j + 1]);
                            }
                            if (ps.vb == 0 && hc == 0) base[(size_t)kDk * kDv + 64 * ps.a + row] = dp;
                        }
                    } else if (ps.c == N - 1 && p.final_state != nullptr && 64 * ps.a + row < p.Dk) {
                        // the sequence's final state [Dk][Dv] (padded channels and columns stay behind)
                        const int col0 = 64 * ps.vb + ch0;
                        ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(p.final_state + ((size_t)ps.bh * p.Dk + 64 * ps.a + row) * p.Dv + col0);
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (col0 + 4 * j < p.Dv) dst[j] = make_ulonglong2(S[2 * j], S[2 * j + 1]);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars[BAR_PURDY + bb]);  // U(c) drained: counts for chunk c + 2
                    if constexpr (NH == 2 && !kHalfSum) {  // the other key half comes next
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const f2 t = S[j];
                            S[j] = So[j];
                            So[j] = t;
                        }
                        const float t = dp;
                        dp = dpo;
                        dpo = t;
                    }
                }
                if (!kSum && !kGenOut && c >= nh && c % nh == 0) {
                    // outputs of the real chunk whose last key half is c-1
                    const int co = c - 1, ob = (co / nh) & 1;
                    const bool fail = !mbar_wait(&bars[BAR_OFULL + (co & 1)], (co >> 1) & 1, abort_flag, limit);
                    if (__any_sync(0xffffffffu, fail)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    uint32_t ow[16];  // the row's 32 outputs packed in pairs
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        uint32_t r[16];
                        tmem_ld_16x32bx2_x16(tmem + lane_base + kColO + ob * 64 + 16 * hf, r);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 8; ++j) ow[8 * hf + j] = Elem<E>::pack(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
                    }
                    tc_fence_before();
                    const int b = fdiv(po.bh, p.fd_H), h = po.bh - b * p.H;
                    const int t = walk_token(p.order, p.T, p.fd_gh, p.grid_w, chunk_w0(p.order, p.T, po.c) + row);
                    store_row<E, NH == 1 || MODE == kFull>(p, ow, b, h, t, 64 * po.vb + ch0);
                }
            }
            if (kBal && piece == 0 && b_chi > 0 && named_barrier_or(3, 128, !ok)) ok = false;
            if (kBal && piece == 0 && b_chi > 0 && ok) {
                // the state at the end of the head run -> the next CTA
                ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(p.summary + (size_t)blockIdx.x * kD * kD + (size_t)row * kD + ch0);
#pragma unroll
                for (int j = 0; j < 8; ++j) dst[j] = make_ulonglong2(S[2 * j], S[2 * j + 1]);
                // the epi's four warps wrote their rows; one thread fences (for them all, after the
                // barrier) and sets the flag, so only its warp waits for its stores in flight
                named_barrier_sync(3, 128);
                if (threadIdx.x == kEpi0 * 32) {
                    __threadfence();
                    *reinterpret_cast<volatile unsigned long long *>(p.flags + blockIdx.x) = p.epoch;
                }
            }
        }
        if (!ok) record_timeout(abort_flag);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// Test hook: launched between a split's passes, it stands for a summary pass that takes longer than the
// limit of the bounded waits: the output pass starts while it runs and waits for it.
__global__ void slow_grid_kernel(unsigned long long ns) {
    pdl_launch_dependents();
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < ns) __nanosleep(1000);
}

// ---------------------------------------------------------------- host side
PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaDriverEntryPointQueryResult q;
        void *f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    });
    return fn;
}

// Row orders: dims (D, H, T, 1, B), box (64, 1, rows, 1, 1).
// Column orders: dims (D, H, W, Hg, B), box (64, 1, 1, rows, 1).
// D is the tensor's row width (Dk or Dv); a box covers 64 channels at x = 0 or 64.
// L2 promotion of 128 bytes, the width of a box row: with 256 bytes every row also fetched
// the neighbouring head's piece of the token row, which the balanced schedule reads much
// later, so DRAM reads rose to 1.38x the input bytes (batched 40x40, H = 12, B = 32: 128-byte
// promotion 1.02x faster there, equal on the other workloads).
bool encode_map(CUtensorMap *m, const void *ptr, const Problem &p, int width, int rows) {
    auto enc = get_encode();
    if (!enc) return false;
    const cuuint64_t es = 2, D = static_cast<cuuint64_t>(width);
    const bool col = (p.order >> 1) != 0;
    cuuint64_t dims[5] = {D, (cuuint64_t)p.H, 0, 0, (cuuint64_t)p.B};
    cuuint64_t strides[4] = {D * es, (cuuint64_t)p.H * D * es, 0, (cuuint64_t)p.T * p.H * D * es};
    cuuint32_t box[5] = {64, 1, 1, 1, 1}, estr[5] = {1, 1, 1, 1, 1};
    if (!col) {
        dims[2] = (cuuint64_t)p.T;
        dims[3] = 1;
        strides[2] = (cuuint64_t)p.T * p.H * D * es;
        box[2] = (cuuint32_t)rows;
    } else {
        dims[2] = (cuuint64_t)p.grid_w;
        dims[3] = (cuuint64_t)p.grid_h;
        strides[2] = (cuuint64_t)p.grid_w * p.H * D * es;
        box[3] = (cuuint32_t)rows;
    }
    const CUtensorMapDataType dt = p.dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    return enc(m, dt, 5, const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

PFN_cuTensorMapEncodeIm2col_v12000 get_encode_im2col() {
    static PFN_cuTensorMapEncodeIm2col_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaDriverEntryPointQueryResult q;
        void *f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeIm2col", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeIm2col_v12000>(f);
    });
    return fn;
}

// Column orders' walk map: the tensor [B][T][H][D] (T = Hg x W tokens, row-major) seen as the
// im2col dims (D, Hg, W, H, B), grid rows fastest: an im2col load of 64 pixels from (y, x, h, b)
// walks down column x and on into the next columns, exactly the column scan.  64 channels per
// pixel at c0 = 0 or 64 (channels past D load as zero); no filter window (all corners 0).
bool encode_col_map(CUtensorMap *m, const void *ptr, const Problem &p, int H, int width) {
    auto enc = get_encode_im2col();
    if (!enc) return false;
    const cuuint64_t es = 2, D = static_cast<cuuint64_t>(width);
    cuuint64_t dims[5] = {D, (cuuint64_t)p.grid_h, (cuuint64_t)p.grid_w, (cuuint64_t)H, (cuuint64_t)p.B};
    cuuint64_t strides[4] = {(cuuint64_t)p.grid_w * H * D * es, (cuuint64_t)H * D * es, D * es,
                             (cuuint64_t)p.T * H * D * es};
    int lower[3] = {0, 0, 0}, upper[3] = {0, 0, 0};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    const CUtensorMapDataType dt = p.dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    return enc(m, dt, 5, const_cast<void *>(ptr), dims, strides, lower, upper, 64, kC, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Gate producer: W2 [H][r][Dk] as dims (Dk, r, H, 1, 1), box (64 channels, r rows): one head's
// block lands as r rows of 128 bytes (SW128, MN-major B of Z = a W2); channels past Dk load as 0.
bool encode_w2_map(CUtensorMap *m, const void *w2, int H, int Dk, int dtype) {
    auto enc = get_encode();
    if (!enc) return false;
    const cuuint64_t es = 2;
    cuuint64_t dims[5] = {(cuuint64_t)Dk, (cuuint64_t)kRank, (cuuint64_t)H, 1, 1};
    cuuint64_t strides[4] = {(cuuint64_t)Dk * es, (cuuint64_t)kRank * Dk * es, (cuuint64_t)H * kRank * Dk * es,
                             (cuuint64_t)H * kRank * Dk * es};
    cuuint32_t box[5] = {64, (cuuint32_t)kRank, 1, 1, 1}, estr[5] = {1, 1, 1, 1, 1};
    const CUtensorMapDataType dt = dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    return enc(m, dt, 5, const_cast<void *>(w2), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Encoded maps are cached per (pointers, shape, order, dtype): a repeated call
// reuses them instead of encoding the maps again.
struct MapKey {
    const void *ptr[kTensors];
    int B, H, grid_h, grid_w, order, dtype, Dk, Dv;
    bool operator==(const MapKey &o) const { return std::memcmp(this, &o, sizeof(MapKey)) == 0; }
};
struct MapEntry {
    MapKey key;
    CUtensorMap maps[kTensors][kHeights];
    CUtensorMap cmaps[kTensors];  // column orders only
};
std::mutex g_map_mutex;
std::list<MapEntry> g_map_cache;  // most recent first
constexpr size_t kMapCacheSize = 32;

bool get_maps(const Problem &p, CUtensorMap (&out)[kTensors][kHeights], CUtensorMap (&cout)[kTensors]) {
    MapKey key;
    std::memset(&key, 0, sizeof(key));
    key.ptr[T_Q] = p.q;
    key.ptr[T_K] = p.k;
    key.ptr[T_V] = p.v;
    key.ptr[T_G] = p.g;
    key.B = p.B;
    key.H = p.H;
    key.grid_h = p.grid_h;
    key.grid_w = p.grid_w;
    key.order = p.order;
    key.dtype = p.dtype;
    key.Dk = p.Dk;
    key.Dv = p.Dv;
    std::lock_guard<std::mutex> lock(g_map_mutex);
    for (auto it = g_map_cache.begin(); it != g_map_cache.end(); ++it) {
        if (it->key == key) {
            std::memcpy(out, it->maps, sizeof(out));
            std::memcpy(cout, it->cmaps, sizeof(cout));
            g_map_cache.splice(g_map_cache.begin(), g_map_cache, it);
            return true;
        }
    }
    MapEntry e;
    e.key = key;
    // row orders load one box height only (60 encodings took 12 us of a first call)
    const bool col = (p.order >> 1) != 0;
    std::memset(e.maps, 0, sizeof(e.maps));
    for (int t = 0; t < kTensors; ++t)
        for (int hi = col ? 0 : kHeights - 1; hi < kHeights; ++hi)
            if (!encode_map(&e.maps[t][hi], key.ptr[t], p, t == T_V ? p.Dv : p.Dk, box_height(hi))) return false;
    std::memset(e.cmaps, 0, sizeof(e.cmaps));
    if (col)
        for (int t = 0; t < kTensors; ++t)
            if (!encode_col_map(&e.cmaps[t], key.ptr[t], p, p.H, t == T_V ? p.Dv : p.Dk)) return false;
    std::memcpy(out, e.maps, sizeof(out));
    std::memcpy(cout, e.cmaps, sizeof(cout));
    g_map_cache.push_front(e);
    if (g_map_cache.size() > kMapCacheSize) g_map_cache.pop_back();
    return true;
}

template <typename E, int NH, int NV, int MODE, bool GENOUT = false, bool GP = false, bool GATED = false>
cudaError_t launch_kernel(dim3 grid, const TcParams &tp, cudaStream_t stream, bool pdl = false) {
    // the shared-memory opt-in, once per process and device (setting it again is harmless)
    static std::atomic<unsigned long long> set_on_devices(0);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(set_on_devices.load(std::memory_order_relaxed) & bit)) {
        e = cudaFuncSetAttribute(gla_tc_kernel<E, NH, NV, MODE, GENOUT, GP, GATED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSmemBytes);
        if (e != cudaSuccess) return e;
        set_on_devices.fetch_or(bit);
    }
    if (MODE == kSplitFull && pdl) {
        // launched right after its summary pass: it may start while that grid runs (programmatic
        // dependent launch) and waits for it before it reads the summaries
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid;
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmemBytes;
        cfg.stream = stream;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, gla_tc_kernel<E, NH, NV, MODE, GENOUT, GP, GATED>, tp);
    }
    gla_tc_kernel<E, NH, NV, MODE, GENOUT, GP, GATED><<<grid, kThreads, kSmemBytes, stream>>>(tp);
    return cudaSuccess;
}

// One instantiation per (element type, key halves, value slices, pass).
// gen_out: outputs stored by the gen warpgroups (fp16, one key half, outputs only)
template <typename E, int MODE>
cudaError_t launch_shape(dim3 grid, const TcParams &tp, cudaStream_t stream, bool gen_out = false, bool pdl = false) {
    if constexpr (std::is_same<E, __half>::value && MODE != kSummary) {
        if (gen_out && tp.nh == 1)
            return tp.nv == 1 ? launch_kernel<E, 1, 1, MODE, true>(grid, tp, stream, pdl)
                              : launch_kernel<E, 1, 2, MODE, true>(grid, tp, stream, pdl);
    }
    if (tp.nh == 1)
        return tp.nv == 1 ? launch_kernel<E, 1, 1, MODE>(grid, tp, stream, pdl)
                          : launch_kernel<E, 1, 2, MODE>(grid, tp, stream, pdl);
    return tp.nv == 1 ? launch_kernel<E, 2, 1, MODE>(grid, tp, stream, pdl)
                      : launch_kernel<E, 2, 2, MODE>(grid, tp, stream, pdl);
}

// kBalanced CTAs wait for their neighbour's hand-off: a cooperative launch guarantees
// that every CTA of the grid is resident at once.
template <typename E, int NV>
cudaError_t launch_balanced(dim3 grid, const TcParams &tp, cudaStream_t stream) {
    static std::atomic<unsigned long long> set_on_devices(0);
    auto kernel = gla_tc_kernel<E, 1, NV, kBalanced, false>;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(set_on_devices.load(std::memory_order_relaxed) & bit)) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
        if (e != cudaSuccess) return e;
        set_on_devices.fetch_or(bit);
    }
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, tp);
}

// Launch epochs of the balanced schedule: nonzero and never repeated within a process,
// so a flag left by an earlier launch (or garbage in a fresh workspace) is not taken for
// this launch's hand-off; flags are also cleared once read, which keeps graph replays of
// one captured launch correct.
unsigned long long next_epoch() {
    static std::atomic<unsigned long long> ctr(
        (static_cast<unsigned long long>(std::chrono::steady_clock::now().time_since_epoch().count()) << 16) | 1ull);
    return ctr.fetch_add(2ull);  // odd, so never 0
}

// Key channels and value columns are processed in 64-wide halves and slices; a
// narrower last one is zero-padded by the TMA loads (boxes past the tensor's row).
int pad64(int d) { return (d + 63) / 64 * 64; }

// Segments per sequence.  A launch whose work units fill fewer than half of the
// SMs splits every sequence into segments of `len` chunks, so that the split
// launch still fits one wave (units x ceil(N / len) <= SMs).  The split's critical
// path is the last segment: `len` chunks in each of the two passes, plus the fold
// of the nseg - 1 earlier summaries into its start state, with several summaries'
// loads in flight.  A graph-replayed sweep of every length on a GB300, of an earlier
// kernel with the fold before the first chunk (batch-1 and small-batch shapes, 64 <= N <= 256
// chunks), fitted about 1.95 us per chunk of length against 0.13 us per segment, so the
// length minimises 15 len + ceil(N / len), at least kMinSegChunks.  (With the present kernels
// two chunks of both passes take 4.0 us and a fold of 12 summaries 2.7; the constants were
// not fitted again.)  Sequences of at most kMaxUnsplitChunks chunks stay whole (6 chunks: 8.9
// us split; 5 chunks: 9.4 us whole and 9.0 split in fp16, 10.0 and 9.4 in bf16, so the line
// could lie one lower now; with the earlier kernels 11.4 and 13.4).
// The last segment may be shorter than the others: its chunks past the sequence
// load as zeros (no key, decay 1), so they leave the state unchanged, and their
// outputs are not stored.
struct Split {
    int nseg;  // segments per sequence (1: no split)
    int len;   // chunks per segment
};

Split choose_split(const Problem &p, int n_sm) {
    const long long N = (p.T + kC - 1) / kC;
    const long long units = (long long)p.B * p.H * (pad64(p.Dv) / 64);
    const Split none{1, static_cast<int>(N)};
    if (units * 2 > n_sm || N <= kMaxUnsplitChunks) return none;
    Split best = none;
    long long best_cost = -1;
    for (long long L = kMinSegChunks; L < N; ++L) {
        const long long d = (N + L - 1) / L;
        if (units * d > n_sm) continue;
        const long long cost = 15 * L + d;
        if (best_cost < 0 || cost < best_cost) {
            best = Split{static_cast<int>(d), static_cast<int>(L)};
            best_cost = cost;
        }
    }
    return best;
}

// Balanced ranges (one key half, unsplit): when the units are more than the SMs and a
// round-robin deal would take at least 1.1 times the chunks per CTA of an even split,
// every CTA takes an equal contiguous range of chunks instead.  Measured on a GB300
// (graph-replayed, interleaved, against whole units): B = 32, H = 12, 40 x 40 (384 units,
// ratio 1.19) 1.10x in bf16 and 1.05x in fp16; B = 16, H = 12, 80 x 80 (192 units, ratio
// 1.58) 1.52x; B = 24 (288 units, ratio 1.06) 0.98x and B = 38 (456 units, ratio 1.00)
// 0.96x, hence the threshold.  The balanced kernel costs about 6 % a chunk more than the
// round-robin one (the hand-offs and the longer decode).
bool choose_balanced(const Problem &p, int n_sm) {
    if (pad64(p.Dk) != 64 || n_sm < 1) return false;
    const long long units = (long long)p.B * p.H * (pad64(p.Dv) / 64);
    if (units <= n_sm) return false;
    if (units * ((p.T + kC - 1) / kC) > 0x7fffffffLL) return false;  // the decode's flattened chunk index is an int
    const long long waves = (units + n_sm - 1) / n_sm;
    return waves * n_sm * 10 >= units * 11;  // ceil(U / SMs) >= 1.1 U / SMs
}

// hand-off states ([64][64] fp32 per CTA) and flags (one 64-bit word per CTA)
size_t handoff_bytes(int n_sm) {
    return (size_t)n_sm * 64 * 64 * sizeof(float) + (size_t)n_sm * sizeof(unsigned long long);
}

size_t summary_bytes(const Problem &p, int nseg) {
    if (nseg <= 1) return 0;
    return (size_t)p.B * p.H * (nseg - 1) * ((size_t)pad64(p.Dk) * pad64(p.Dv) + pad64(p.Dk)) * sizeof(float);
}

}  // namespace

cudaError_t sm_count(int *n_sm) {  // cached per device
    static std::atomic<int> cache[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) {
        const int v = cache[dev].load(std::memory_order_relaxed);
        if (v > 0) {
            *n_sm = v;
            return cudaSuccess;
        }
    }
    e = cudaDeviceGetAttribute(n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && dev >= 0 && dev < 64) cache[dev].store(*n_sm, std::memory_order_relaxed);
    return e;
}

int tc_chunk_boxes(int order, int T, int grid_h, int grid_w, int c, int *boxes, int cap) {
    int n = 0;
    chunk_load_boxes(order, T, make_fastdiv(grid_h), grid_w, c, [&](int hi, int row, int c2, int c3) {
        if (n < cap) {
            boxes[4 * n + 0] = box_height(hi);
            boxes[4 * n + 1] = row;
            boxes[4 * n + 2] = c2;
            boxes[4 * n + 3] = c3;
        }
        ++n;
    });
    return n;
}

int tc_balanced_walk(int n_units, int N, int grid, int cta, int *entries, int cap, int *head) {
    const BalRange r = bal_range(N, n_units, cta, grid);
    const FastDiv fn = make_fastdiv(N);
    for (int v = 0; v < r.G && v < cap; ++v) {
        const StreamPos ps = stream_pos_bal(v, N, 0, r.base_head, r.base_full, r.base_tail, r.c_hi, r.t0, fn);
        entries[4 * v + 0] = ps.bh;  // with one value slice per unit, the unit itself
        entries[4 * v + 1] = ps.c;
        entries[4 * v + 2] = ps.start ? 1 : 0;
        entries[4 * v + 3] = ps.hin ? 1 : 0;
    }
    *head = r.c_hi;
    return r.G;
}

int tc_chunk_walk(int order, int T, int grid_h, int c, int *x0, int *y0) {
    return chunk_walk_start(order, T, make_fastdiv(grid_h), c, x0, y0) ? 1 : 0;
}

void tc_split_plan(const Problem &p, int n_sm, int *nseg, int *seg_len) {
    const Split sp = choose_split(p, n_sm);
    *nseg = sp.nseg;
    *seg_len = sp.len;
}

size_t tc_workspace_bytes(const Problem &p) {
    int n_sm = 0;
    if (sm_count(&n_sm) != cudaSuccess) return 0;
    const int nseg = choose_split(p, n_sm).nseg;
    if (nseg > 1) return summary_bytes(p, nseg);
    return choose_balanced(p, n_sm) ? handoff_bytes(n_sm) : 0;
}

int tc_balanced_plan(const Problem &p, int n_sm) { return choose_split(p, n_sm).nseg == 1 && choose_balanced(p, n_sm); }

bool tc_supported(const Problem &p) {
    if (p.dtype != 1 && p.dtype != 2) return false;       // fp16 / bf16 operands only
    // rows of 16-byte multiples (TMA strides); up to two 64-wide halves / slices
    if (p.Dk % 8 != 0 || p.Dv % 8 != 0 || p.Dk > 128 || p.Dv > 128) return false;
    if (p.T > (1 << 30)) return false;
    return get_encode() != nullptr;
}

cudaError_t launch_tc(const Problem &p, cudaStream_t stream, void *workspace, size_t workspace_bytes, Ran *ran,
                      const Gate *gate, bool *gate_fused) {
    if (gate_fused) *gate_fused = false;
    TcParams tp;
    if (!get_maps(p, tp.maps, tp.cmaps)) return cudaErrorInvalidValue;
    int n_sm = 0;
    cudaError_t e = sm_count(&n_sm);
    if (e != cudaSuccess) return e;
    tp.out = p.out;
    tp.final_state = p.final_state;
    tp.H = p.H;
    tp.out_row = static_cast<unsigned long long>(p.H) * p.Dv;
    tp.grid_h = p.grid_h;
    tp.fd_H = make_fastdiv(p.H);
    tp.fd_gh = make_fastdiv(p.grid_h);
    tp.grid_w = p.grid_w;
    tp.order = p.order;
    tp.T = static_cast<int>(p.T);
    tp.n_chunks = static_cast<int>((p.T + kC - 1) / kC);
    tp.Dk = p.Dk;
    tp.Dv = p.Dv;
    tp.nh = pad64(p.Dk) / 64;
    tp.nv = pad64(p.Dv) / 64;
    Split sp = choose_split(p, n_sm);
    Ran r;
    const bool bal = choose_balanced(p, n_sm);
    r.planned = sp.nseg > 1 ? kRanTcSplit : (bal ? kRanTcBalanced : kRanTc);
    r.ran = kRanTc;
    if (sp.nseg > 1 && (workspace == nullptr || workspace_bytes < summary_bytes(p, sp.nseg)))
        sp = Split{1, tp.n_chunks};
    if (sp.nseg > 1) r.ran = kRanTcSplit;
    const int nseg = sp.nseg;
    tp.nseg = nseg;
    tp.seg_len = sp.len;
    tp.fd_L = make_fastdiv(sp.len);
    tp.summary = static_cast<float *>(workspace);
    tp.wait_limit = kWaitLimitNs + kSummaryChunkNs * static_cast<unsigned long long>(sp.len);
    tp.flags = nullptr;
    tp.epoch = 0;
    // test hooks: 1, the timeout path (no fault: the data of one chunk simply never arrives); 2, a slow
    // grid between a split's passes
    const char *drop = std::getenv("GTR_GLA_TEST_DROP_LOAD");
    tp.drop_load = (drop != nullptr && drop[0] == '1') ? 1 : 0;
    const int seqs = static_cast<int>(p.B * p.H) * tp.nv;  // (sequence, value slice) pairs
    const bool half = p.dtype == 1;
    // persistent: one CTA per SM, each walking its share of the work units
    unsigned sum_ctas = 0;
    if (nseg > 1) {  // pass 1: end state from zero and total decay of segments 0 .. nseg-2
        // (two key halves: a unit is one half with every value slice)
        tp.nsu = nseg - 1;
        tp.fd_nsu = make_fastdiv(tp.nsu);
        tp.n_units = (tp.nh == 2 ? 2 * static_cast<int>(p.B * p.H) : seqs) * tp.nsu;
        tp.fd_per = make_fastdiv(sp.len);
        const dim3 grid(static_cast<unsigned>(tp.n_units < n_sm ? tp.n_units : n_sm));
        sum_ctas = grid.x;
        e = half ? launch_shape<__half, kSummary>(grid, tp, stream) : launch_shape<__nv_bfloat16, kSummary>(grid, tp, stream);
        if (e != cudaSuccess) return e;
        if (drop != nullptr && drop[0] == '2') slow_grid_kernel<<<1, 32, 0, stream>>>(kWaitLimitNs + kSummaryChunkNs / 2 * sp.len);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    tp.nsu = nseg;
    tp.fd_nsu = make_fastdiv(nseg);
    tp.n_units = seqs * nseg;
    tp.fd_per = make_fastdiv(sp.len * tp.nh);
    if (nseg == 1 && bal && workspace != nullptr && workspace_bytes >= handoff_bytes(n_sm)) {
        // equal contiguous chunk ranges, one CTA per SM
        r.ran = kRanTcBalanced;
        if (ran) *ran = r;
        tp.flags = reinterpret_cast<unsigned long long *>(static_cast<char *>(workspace) + (size_t)n_sm * 64 * 64 * sizeof(float));
        tp.epoch = next_epoch();
        tp.bal_n = make_fastdiv(tp.n_chunks);
        const dim3 bgrid(static_cast<unsigned>(n_sm));
        if (half)
            e = tp.nv == 1 ? launch_balanced<__half, 1>(bgrid, tp, stream) : launch_balanced<__half, 2>(bgrid, tp, stream);
        else
            e = tp.nv == 1 ? launch_balanced<__nv_bfloat16, 1>(bgrid, tp, stream)
                           : launch_balanced<__nv_bfloat16, 2>(bgrid, tp, stream);
        if (e != cudaSuccess) return e;
        return cudaGetLastError();
    }
    if (ran) *ran = r;
    // output gate fused into the stores: one key half and one value slice (a row's Dv outputs in
    // one thread pair), outputs stored by the gen warpgroups, for launches of few sequences (at
    // most half as many units as SMs), where it saves a launch: measured on a GB300 (graph
    // replays, interleaved) 3.5 % faster at B = 1, H = 6, 40 x 40, but 1.14-1.26x slower than
    // the separate gate kernel at B = 32, H = 12, 40 x 40 and B = 8, H = 16, 80 x 80, where the
    // gate's work lands on the gen warpgroups' share of the critical chain
    const bool fuse = gate != nullptr && tp.nh == 1 && tp.nv == 1 && 2 * seqs <= n_sm;
    if (fuse) {
        tp.gate_r = gate->r;
        tp.gate_w = gate->w;
        tp.gate_eps = gate->eps;
        if (gate_fused) *gate_fused = true;
    }
    // the fewest CTAs that keep the busiest one's unit count: equal shares, and no SM works
    // on a short share while the others finish (measured on a GB300: B = 32, H = 12, 40 x 40,
    // bf16, 384 units on 128 CTAs instead of 152 ran 3 % faster, the same at fp16)
    const int per_cta = (tp.n_units + n_sm - 1) / n_sm;
    const dim3 grid(static_cast<unsigned>((tp.n_units + per_cta - 1) / per_cta));
    // outputs from the gen warpgroups: fp16 launches of at most one wave (GB300, graph replays, stored by
    // the epi / here: 6,400 tokens, B = 8, H = 16, strong decays 149.6 / 148.0 us, mild 106.4 / 104.4; 64 heads
    // of 64 x 64 80.9 / 79.5; 12 heads, B = 12, 40 x 40 32.5 / 32.1; six heads of 24 x 16 9.25 / 8.88.  With
    // several units per CTA, or bf16, the epi storing them was faster, measured with earlier kernels)
    const bool gen_out = half && tp.n_units <= n_sm;
    // The output pass of a split starts while its summary pass runs (its CTAs start once every summary
    // CTA has).  One key half: always; CTAs load and prepare their first chunks on SMs as they free up
    // (GB300, graph replays, pass sizes in CTAs: 96 + 144, B = 4, H = 12, 40 x 40 27.8 -> 26.2 us; 90 + 96
    // 15.4 -> 14.4; 24 heads of 56 x 56 28.1 -> 26.9; 128 x 128 with 2 heads 26.4 -> 25.5).  Two key halves,
    // whose CTAs only set up before they wait: when both fit on the SMs at once (90 + 93 CTAs of 44 x 44
    // 22.0 us against 22.9, 96 + 128 of 128 x 128 the same).
    const bool pdl = nseg > 1 && (tp.nh == 1 || sum_ctas + grid.x <= static_cast<unsigned>(n_sm));
    if (fuse) {
        if (nseg > 1)
            e = half ? launch_kernel<__half, 1, 1, kSplitFull, true, false, true>(grid, tp, stream, pdl)
                     : launch_kernel<__nv_bfloat16, 1, 1, kSplitFull, true, false, true>(grid, tp, stream, pdl);
        else
            e = half ? launch_kernel<__half, 1, 1, kFull, true, false, true>(grid, tp, stream)
                     : launch_kernel<__nv_bfloat16, 1, 1, kFull, true, false, true>(grid, tp, stream);
        if (e != cudaSuccess) return e;
        return cudaGetLastError();
    }
    if (nseg > 1)
        e = half ? launch_shape<__half, kSplitFull>(grid, tp, stream, gen_out, pdl)
                 : launch_shape<__nv_bfloat16, kSplitFull>(grid, tp, stream, false, pdl);
    else
        e = half ? launch_shape<__half, kFull>(grid, tp, stream, gen_out)
                 : launch_shape<__nv_bfloat16, kFull>(grid, tp, stream);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

bool tc_gate_supported(const Problem &p, int rank) {
    // one 64-channel key half, the paper's rank, and units of at least four chunks (the W2 block
    // of a unit is double-buffered by unit parity, see the producer)
    return tc_supported(p) && p.Dk <= 64 && rank == kRank && p.T > 3 * kC;
}

cudaError_t launch_tc_gate(const Problem &p, const GateSource &gs, cudaStream_t stream, Ran *ran) {
    if (!tc_gate_supported(p, kRank) || !(gs.tau > 0.f)) return cudaErrorInvalidValue;
    TcParams tp;
    std::memset(&tp, 0, sizeof(tp));
    // q, k and v as in the plain schedule; the gate tiles' maps then load the projection a
    // ([B, T, r] as a one-head tensor of width r, boxes 64 elements wide: the row's other 48
    // elements are zero-filled, so the a tile has 128-byte rows like the other tiles)
    Problem pq = p;
    pq.g = p.q;
    if (!get_maps(pq, tp.maps, tp.cmaps)) return cudaErrorInvalidValue;
    Problem pa = p;
    pa.H = 1;
    for (int hi = (p.order >> 1) != 0 ? 0 : kHeights - 1; hi < kHeights; ++hi)
        if (!encode_map(&tp.maps[T_G][hi], gs.a_low, pa, kRank, box_height(hi))) return cudaErrorInvalidValue;
    if ((p.order >> 1) != 0 && !encode_col_map(&tp.cmaps[T_G], gs.a_low, p, 1, kRank)) return cudaErrorInvalidValue;
    if (!encode_w2_map(&tp.w2map, gs.w2, p.H, p.Dk, p.dtype)) return cudaErrorInvalidValue;
    tp.gbias = gs.bias;
    tp.tau_inv = 1.f / gs.tau;
    int n_sm = 0;
    cudaError_t e = sm_count(&n_sm);
    if (e != cudaSuccess) return e;
    tp.out = p.out;
    tp.final_state = p.final_state;
    tp.H = p.H;
    tp.out_row = static_cast<unsigned long long>(p.H) * p.Dv;
    tp.grid_h = p.grid_h;
    tp.fd_H = make_fastdiv(p.H);
    tp.fd_gh = make_fastdiv(p.grid_h);
    tp.grid_w = p.grid_w;
    tp.order = p.order;
    tp.T = static_cast<int>(p.T);
    tp.n_chunks = static_cast<int>((p.T + kC - 1) / kC);
    tp.Dk = p.Dk;
    tp.Dv = p.Dv;
    tp.nh = 1;
    tp.nv = pad64(p.Dv) / 64;
    tp.nseg = 1;
    tp.nsu = 1;
    tp.seg_len = tp.n_chunks;
    tp.fd_nsu = make_fastdiv(1);
    tp.fd_L = make_fastdiv(tp.n_chunks);
    tp.fd_per = make_fastdiv(tp.n_chunks);
    const char *drop = std::getenv("GTR_GLA_TEST_DROP_LOAD");
    tp.drop_load = (drop != nullptr && drop[0] == '1') ? 1 : 0;
    tp.n_units = static_cast<int>(p.B * p.H) * tp.nv;
    if (ran) *ran = Ran{kRanTc, kRanTc};
    const int per_cta = (tp.n_units + n_sm - 1) / n_sm;
    const dim3 grid(static_cast<unsigned>((tp.n_units + per_cta - 1) / per_cta));
    const bool gen_out = p.dtype == 1 && tp.n_units <= n_sm;  // as the plain schedule
    if (p.dtype == 1) {
        if (gen_out)
            e = tp.nv == 1 ? launch_kernel<__half, 1, 1, kFull, true, true>(grid, tp, stream)
                           : launch_kernel<__half, 1, 2, kFull, true, true>(grid, tp, stream);
        else
            e = tp.nv == 1 ? launch_kernel<__half, 1, 1, kFull, false, true>(grid, tp, stream)
                           : launch_kernel<__half, 1, 2, kFull, false, true>(grid, tp, stream);
    } else {
        e = tp.nv == 1 ? launch_kernel<__nv_bfloat16, 1, 1, kFull, false, true>(grid, tp, stream)
                       : launch_kernel<__nv_bfloat16, 1, 2, kFull, false, true>(grid, tp, stream);
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

void *tensor_map_encoder() { return reinterpret_cast<void *>(get_encode()); }

cudaError_t read_and_clear_device_status(unsigned int *status) {
    cudaError_t e = cudaMemcpyFromSymbol(status, g_device_status, sizeof(unsigned int));
    if (e != cudaSuccess) return e;
    const unsigned int zero = 0;
    return cudaMemcpyToSymbol(g_device_status, &zero, sizeof(unsigned int));
}

}  // namespace gtr
