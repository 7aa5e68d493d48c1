// gla_simt.cu -- plain fp32 CUDA-core token recurrence.
//
// Sec. 3.1 ("Key-only gated recurrence"): S_t = Diag(gamma_t) S_{t-1} + k_t^T v_t,
// o_t = q_t S_t, walked token by token along the scan order of Sec. 3.1
// ("Directional scanning").  This is the float32 path (the tensor-core schedule
// cannot hold a 1e-5 relative error) and the path for shapes the tensor-core
// schedule does not take.
//
// What bounds it: three fp32 operations per state element and token (k v, the decayed
// add, the readout), 3 Dk Dv per token-head, on 128 lanes an SM (12 us for 38,400
// token-heads at Dk = Dv = 64; HBM needs 7), and below about 100 sequences the serial
// chain of tokens.
//
// Mapping: a group of compute threads walks one sequence, or one segment of it, for 64
// value columns.  A thread owns an 8 x 8 tile of S in registers as packed pairs of rows
// (fma.rn.f32x2: two IEEE fp32 operations per instruction), so a token costs it 8
// shared-memory vector reads for 96 packed operations (4 columns a thread instead of 8
// read 1.6x the bytes and were bound by shared memory).  As many helper threads load and
// stage the next eight tokens meanwhile (gamma = e^g formed once per element) and add and
// store the last eight tokens' partial readouts, one per row group.  The permutation is
// applied when loading (gather) and when storing o_t (scatter back to the spatial position).
//
// Few sequences leave most SMs idle, and a sequence is a serial chain of tokens.  Such
// launches cut every sequence into segments walked by the CTAs of one thread-block
// cluster (choose_cluster): each group first runs its segment from zero (k, v and gamma
// only) and leaves the end state and the total decay in its shared memory; then the
// earlier segments' are folded (S_start = sum_s' (prod_{s' < s''} D_s'') S_end(s'), Eq.
// chunk_boundary_main across segments) through distributed shared memory and the segment
// is walked again with the outputs.  One launch and no workspace: calls under stream
// capture, on several streams or with no scratch run the same way.
//
// Narrow values, few key channels and short sequences would leave most of the tiles
// empty: whole sequences of those take the kernel of 16 columns a CTA (narrow_columns).
//
// Measured on a GB300 (graph replays, fp32, Dk = Dv = 64), against one CTA of 256 threads
// per 16 columns walking whole sequences: 24 sequences of 1,600 tokens 63 us (440 before),
// 2 of 256 tokens 14 us (43 before).  Up to 32 key channels the helper and compute roles
// spill (36 to 60 bytes of stores a thread, up to 64 channels 4).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <atomic>

#include "f32x2.cuh"
#include "fastdiv.cuh"
#include "gla_internal.h"

namespace gtr {
namespace {

constexpr int kTok = 8;        // tokens staged per block
constexpr int kCols = 64;      // value columns per CTA
constexpr int kVec = kCols / 4;   // staged float4s of v per token
constexpr int kMaxCluster = 16;  // CTAs of a cluster (above 8 needs the non-portable opt-in)

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__half x) { return __half2float(x); }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }

template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ __half from_f32<__half>(float x) { return __float2half_rn(x); }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) {
    return __float2bfloat16_rn(x);
}

// Thread-block cluster: arrive (release) and wait (acquire) on its barrier, and a generic
// pointer to the same shared-memory address in another of its CTAs.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ const float *cluster_peer(const float *p, int rank) {
    unsigned long long r;
    asm("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(reinterpret_cast<unsigned long long>(p)), "r"(rank));
    return reinterpret_cast<const float *>(r);
}

struct SimtParams {
    Problem p;
    FastDiv fd_H, fd_gh;
    int n_seqs;
    int nseg;           // segments per sequence: 1, or the groups of a whole cluster
    long long seg_len;  // tokens per segment, a multiple of kTok (the last ones may be short or empty)
};

// Spatial token visited at scan position s (Sec. 3.1 "Directional scanning").
__device__ __forceinline__ int scan_token(const SimtParams &sp, unsigned s) {
    const int u = (sp.p.order & 1) ? static_cast<int>(sp.p.T) - 1 - static_cast<int>(s) : static_cast<int>(s);
    if ((sp.p.order >> 1) == 0) return u;
    const int x = fdiv(u, sp.fd_gh);
    return (u - x * sp.fd_gh.d) * sp.p.grid_w + x;
}

// Four consecutive elements i .. i + 3 of a row of `width`, zeros past its end.  VEC: widths are
// multiples of four (and rows therefore aligned to four elements).
template <typename E, bool VEC>
__device__ __forceinline__ float4 load4(const E *row, int i, int width) {
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (VEC) {
        if (i < width) {
            if constexpr (sizeof(E) == 4) {
                r = *reinterpret_cast<const float4 *>(row + i);
            } else {
                const uint2 w = *reinterpret_cast<const uint2 *>(row + i);
                const E *e = reinterpret_cast<const E *>(&w);
                r = make_float4(to_f32(e[0]), to_f32(e[1]), to_f32(e[2]), to_f32(e[3]));
            }
        }
    } else {
        if (i < width) r.x = to_f32(row[i]);
        if (i + 1 < width) r.y = to_f32(row[i + 1]);
        if (i + 2 < width) r.z = to_f32(row[i + 2]);
        if (i + 3 < width) r.w = to_f32(row[i + 3]);
    }
    return r;
}

__device__ __forceinline__ float gamma_of(float lg) {
    lg = lg < -1.0e4f ? -1.0e4f : lg;  // gamma = 0 below -1e4; NaN stays NaN
    return expf(lg);
}

// A CTA is 4 compute warps and 4 helper warps, in G groups of DKM compute and DKM helper threads;
// each group walks its own sequence or segment.  (A group of two compute warps alone would sit on
// two of the SM's four sub-partitions, and so would every other CTA's.)
//
// Shared memory of a group (floats): two buffers of staged inputs, two of partial readouts (before
// them, in the first, the segment's state), the segment's decay, the spatial tokens of four blocks.
template <int DKM>
struct SimtShape {
    static constexpr int RG = DKM / 8;                    // row groups of 8 rows
    static constexpr int threads = DKM;                   // compute threads of a group: RG x 8 column groups
    static constexpr int G = 128 / threads;
    static constexpr int q = 0, k = kTok * DKM, g = 2 * kTok * DKM, v = 3 * kTok * DKM;
    static constexpr int stage = 3 * kTok * DKM + kTok * kCols;
    static constexpr int po = 2 * stage, po_n = kTok * RG * kCols;  // [kTok][RG][64], or a state [DKM][64]
    static constexpr int decay = po + 2 * po_n;           // [DKM]
    static constexpr int tok = decay + DKM;               // (int)
    static constexpr int group = tok + 4 * kTok;
    static constexpr int bytes = G * group * 4;
    static constexpr int qu = 2;                          // staged float4s of q, k and gamma per helper thread
    static constexpr int vu = kTok * kVec / threads;      // and of v
    static constexpr int cu = threads < kCols ? kCols / threads : 1;  // summary: columns of v per helper thread
    static_assert(kTok == 8 && RG * 8 == threads && qu * threads * 4 == kTok * DKM && po_n == DKM * kCols, "layout");
};

constexpr int kSimtThreads = 256;

template <int DKM, typename E, bool VEC>
__global__ void __launch_bounds__(kSimtThreads, 2) gla_simt_kernel(const __grid_constant__ SimtParams sp) {
    using Sh = SimtShape<DKM>;
    constexpr int RG = Sh::RG, G = Sh::G;
    extern __shared__ __align__(16) float smem[];
    const Problem &p = sp.p;
    const int nseg = sp.nseg;
    // the first four warps compute; the others (helpers) load and stage the next blocks and store
    // the outputs of the last one meanwhile
    const bool helper = threadIdx.x >= kSimtThreads / 2;
    const int ct = threadIdx.x % (kSimtThreads / 2);
    const int grp = ct / Sh::threads, tid = ct % Sh::threads, lane = tid & 31, warp = tid >> 5;
    float *sm = smem + grp * Sh::group;
    const unsigned unit = blockIdx.x * static_cast<unsigned>(G) + grp;  // (sequence, segment)
    const unsigned seq = nseg > 1 ? unit / static_cast<unsigned>(nseg) : unit;
    const bool live = seq < static_cast<unsigned>(sp.n_seqs);
    const int bh = live ? static_cast<int>(seq) : 0, seg = nseg > 1 ? static_cast<int>(unit - seq * nseg) : 0;
    const int b = fdiv(bh, sp.fd_H), h = bh - b * p.H;
    const int c0 = static_cast<int>(blockIdx.y) * kCols;
    // a compute thread's rows are 4 rg + {0..3} of the lower and of the upper half of the rows, its
    // columns 4 cg + {0..3} of the two halves of the columns; a warp covers RG (at most 8) row groups
    constexpr int kRgWarp = RG < 8 ? RG : 8, kCgWarp = 32 / kRgWarp, kCgWarps = 8 / kCgWarp;
    const int rg = lane / kCgWarp + kRgWarp * (warp / kCgWarps), cg = lane % kCgWarp + kCgWarp * (warp % kCgWarps);
    const int Dk = p.Dk, Dv = p.Dv;
    const long long T = p.T;
    // row base of token t: (b T + t) H + h rows of Dk or Dv elements
    const long long row0 = (static_cast<long long>(b) * T) * p.H + h;
    const E *q = static_cast<const E *>(p.q), *k = static_cast<const E *>(p.k);
    const E *v = static_cast<const E *>(p.v), *g = static_cast<const E *>(p.g);
    E *out = static_cast<E *>(p.out);
    auto group_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(2 * Sh::threads) : "memory"); };

    const long long t0l = seg * sp.seg_len, t1l = t0l + sp.seg_len;
    const unsigned t0 = static_cast<unsigned>(t0l < T ? t0l : T);
    const unsigned t1 = !live ? t0 : static_cast<unsigned>(t1l < T ? t1l : T);

    // the last segment's own state is not needed, and an empty one's is zero with decay 1
    const bool want_sum = nseg > 1 && seg < nseg - 1 && t0 < t1;
    const unsigned nblk = (t1 - t0 + kTok - 1) / kTok;
    float *ss = sm + Sh::po, *sd = sm + Sh::decay;     // the group's state and decay (before the outputs)
    float *ps = smem + Sh::po + Sh::po_n;              // the state at the start of the CTA's first segment

    if (helper) {
        // ================================================= helpers (their registers go to the compute warps)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 80;");
        if (want_sum) {
            // a helper thread stages channel tid and (as far as there are any) columns tid, tid + threads
            float rk[kTok], rgm[kTok], rv[Sh::cu][kTok];
            auto load_sum = [&](unsigned s0) {
#pragma unroll
                for (int j = 0; j < kTok; ++j) {
                    rk[j] = rgm[j] = 0.f;
#pragma unroll
                    for (int m = 0; m < Sh::cu; ++m) rv[m][j] = 0.f;
                    if (s0 + j < t1) {
                        const long long row = row0 + static_cast<long long>(scan_token(sp, s0 + j)) * p.H;
                        if (tid < Dk) {
                            rk[j] = to_f32(k[row * Dk + tid]);
                            rgm[j] = to_f32(g[row * Dk + tid]);
                        }
#pragma unroll
                        for (int m = 0; m < Sh::cu; ++m) {
                            const int c = tid + m * Sh::threads;
                            if (c < kCols && c0 + c < Dv) rv[m][j] = to_f32(v[row * Dv + c0 + c]);
                        }
                    }
                }
            };
            auto stage_sum = [&](int buf) {
                float *st = sm + buf * Sh::stage;
                float run = 1.f;
#pragma unroll
                for (int j = kTok - 1; j >= 0; --j) {
                    st[Sh::k + j * DKM + tid] = rk[j] * run;
                    run *= gamma_of(rgm[j]);
                }
                st[Sh::g + tid] = run;
#pragma unroll
                for (int m = 0; m < Sh::cu; ++m)
#pragma unroll
                    for (int j = 0; j < kTok; ++j)
                        if (tid + m * Sh::threads < kCols) st[Sh::v + j * kCols + tid + m * Sh::threads] = rv[m][j];
            };
            load_sum(t0);
            stage_sum(0);
            load_sum(t0 + kTok);  // (zeros past the segment)
            group_sync();
            int buf = 0;
            for (unsigned s0 = t0; s0 < t1; s0 += kTok, buf ^= 1) {
                if (s0 + kTok < t1) {
                    stage_sum(buf ^ 1);
                    load_sum(s0 + 2 * kTok);
                }
                group_sync();
            }
        }
        if (nseg > 1) {
            for (int gi = 0; gi + 1 < G; ++gi) __syncthreads();  // the groups' running states, below
            cluster_arrive();
            cluster_wait();
            // the state at the start of the CTA's first segment, folded from the earlier CTAs' running
            // states (their last group's) from the latest back
            const int rank = seg / G;
            const float *ls = smem + (G - 1) * Sh::group + Sh::po, *ld = smem + (G - 1) * Sh::group + Sh::decay;
            constexpr int kPer = DKM < 64 ? DKM * kVec / (kSimtThreads / 2) : 8;  // float4s of the state at a time
#pragma unroll 1
            for (int u0 = ct; u0 < DKM * kVec; u0 += kPer * (kSimtThreads / 2)) {
                float4 acc[kPer];
                float coef[kPer];
#pragma unroll
                for (int m = 0; m < kPer; ++m) acc[m] = make_float4(0.f, 0.f, 0.f, 0.f), coef[m] = 1.f;
#pragma unroll 1
                for (int s2 = rank - 1; s2 >= 0; --s2) {
                    const float *rs = cluster_peer(ls, s2), *rd = cluster_peer(ld, s2);
#pragma unroll
                    for (int m = 0; m < kPer; ++m) {
                        const int u = u0 + m * (kSimtThreads / 2);
                        const float4 x = *reinterpret_cast<const float4 *>(rs + 4 * u);
                        const float d = rd[u / kVec];
                        acc[m].x = fmaf(coef[m], x.x, acc[m].x);
                        acc[m].y = fmaf(coef[m], x.y, acc[m].y);
                        acc[m].z = fmaf(coef[m], x.z, acc[m].z);
                        acc[m].w = fmaf(coef[m], x.w, acc[m].w);
                        coef[m] *= d;
                    }
                }
#pragma unroll
                for (int m = 0; m < kPer; ++m) *reinterpret_cast<float4 *>(ps + 4 * (u0 + m * (kSimtThreads / 2))) = acc[m];
            }
            cluster_arrive();  // this CTA has read its peers' states
            __syncthreads();   // the compute warps take theirs
        }
        // ---- the tokens with their outputs.  One block's inputs in registers (zeros, gamma = 1
        // past the segment and past Dk, Dv: padding contributes nothing)
        float4 rq[Sh::qu], rk[Sh::qu], rgm[Sh::qu], rv[Sh::vu];
        int rt[Sh::vu];
        auto load_block = [&](unsigned s0) {
#pragma unroll
            for (int m = 0; m < Sh::qu; ++m) {
                const int u = tid + m * Sh::threads, j = u / (DKM / 4), i = 4 * (u % (DKM / 4));
                rq[m] = rk[m] = rgm[m] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (s0 + j < t1) {
                    const long long row = (row0 + static_cast<long long>(scan_token(sp, s0 + j)) * p.H) * Dk;
                    rq[m] = load4<E, VEC>(q + row, i, Dk);
                    rk[m] = load4<E, VEC>(k + row, i, Dk);
                    rgm[m] = load4<E, VEC>(g + row, i, Dk);
                }
            }
#pragma unroll
            for (int m = 0; m < Sh::vu; ++m) {
                const int u = tid + m * Sh::threads, j = u / kVec, i = 4 * (u % kVec);
                rv[m] = make_float4(0.f, 0.f, 0.f, 0.f);
                rt[m] = 0;
                if (s0 + j < t1) {
                    rt[m] = scan_token(sp, s0 + j);
                    rv[m] = load4<E, VEC>(v + (row0 + static_cast<long long>(rt[m]) * p.H) * Dv, c0 + i, Dv);
                }
            }
        };
        auto stage_block = [&](int buf, int tbuf) {
            float *st = sm + buf * Sh::stage;
#pragma unroll
            for (int m = 0; m < Sh::qu; ++m) {
                const int o = 4 * (tid + m * Sh::threads);  // [token][channel]
                *reinterpret_cast<float4 *>(st + Sh::q + o) = rq[m];
                *reinterpret_cast<float4 *>(st + Sh::k + o) = rk[m];
                *reinterpret_cast<float4 *>(st + Sh::g + o) =
                    make_float4(gamma_of(rgm[m].x), gamma_of(rgm[m].y), gamma_of(rgm[m].z), gamma_of(rgm[m].w));
            }
#pragma unroll
            for (int m = 0; m < Sh::vu; ++m) {
                const int u = tid + m * Sh::threads;
                *reinterpret_cast<float4 *>(st + Sh::v + 4 * u) = rv[m];
                if (u % kVec == 0) reinterpret_cast<int *>(sm + Sh::tok)[tbuf * kTok + u / kVec] = rt[m];
            }
        };
        // a block's outputs: sum over the row groups, scattered to the spatial tokens
        auto store_block = [&](unsigned s0, int buf, int tbuf) {
            const float *po = sm + Sh::po + buf * Sh::po_n;
#pragma unroll
            for (int m = 0; m < Sh::vu; ++m) {
                const int u = tid + m * Sh::threads, jv = u / kVec, iv = 4 * (u % kVec);
                if (s0 + jv >= t1 || c0 + iv >= Dv) continue;
                float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int r = 0; r < RG; ++r) {
                    const float4 x = *reinterpret_cast<const float4 *>(po + (jv * RG + r) * kCols + (iv ^ ((r & 1) << 4)));
                    o.x += x.x;
                    o.y += x.y;
                    o.z += x.z;
                    o.w += x.w;
                }
                const int t = reinterpret_cast<const int *>(sm + Sh::tok)[tbuf * kTok + jv];
                E *dst = out + (row0 + static_cast<long long>(t) * p.H) * Dv + c0 + iv;
                if constexpr (VEC) {
                    if constexpr (sizeof(E) == 4) {
                        *reinterpret_cast<float4 *>(dst) = o;
                    } else {
                        uint2 w;
                        E *e = reinterpret_cast<E *>(&w);
                        e[0] = from_f32<E>(o.x);
                        e[1] = from_f32<E>(o.y);
                        e[2] = from_f32<E>(o.z);
                        e[3] = from_f32<E>(o.w);
                        *reinterpret_cast<uint2 *>(dst) = w;
                    }
                } else {
                    dst[0] = from_f32<E>(o.x);
                    if (c0 + iv + 1 < Dv) dst[1] = from_f32<E>(o.y);
                    if (c0 + iv + 2 < Dv) dst[2] = from_f32<E>(o.z);
                    if (c0 + iv + 3 < Dv) dst[3] = from_f32<E>(o.w);
                }
            }
        };
        if (t0 < t1) {
            load_block(t0);
            stage_block(0, 0);
            load_block(t0 + kTok);  // (zeros past the segment)
        }
        if (nseg > 1) {
            cluster_wait();   // the peers have read this CTA's states
            __syncthreads();  // and its own groups theirs: the partial readouts may go there
        }
        if (t0 >= t1) return;
        group_sync();
        for (unsigned n = 0; n <= nblk; ++n) {
            const unsigned s0 = t0 + n * kTok;
            const int buf = static_cast<int>(n & 1);
            if (n > 0) store_block(s0 - kTok, buf ^ 1, static_cast<int>((n - 1) & 3));
            if (n + 1 < nblk) {
                stage_block(buf ^ 1, static_cast<int>((n + 1) & 3));
                load_block(s0 + 2 * kTok);
            }
            group_sync();
        }
        return;
    }

    // ===================================================== compute warps
    asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
    // a thread's operands of token j of a staged block: four pairs of rows, eight columns
    struct Rows {
        f2 r[4];
    };
    struct Cols {
        float4 c[2];
    };
    auto rows_of = [&](const float *base, int j) {
        Rows x;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(base + j * DKM + m * (DKM / 2) + 4 * rg);
            x.r[2 * m] = w.x;
            x.r[2 * m + 1] = w.y;
        }
        return x;
    };
    auto cols_of = [&](const float *base, int j) {
        Cols x;
#pragma unroll
        for (int m = 0; m < 2; ++m) x.c[m] = *reinterpret_cast<const float4 *>(base + j * kCols + m * (kCols / 2) + 4 * cg);
        return x;
    };
    auto spread = [](const Cols &x, f2 (&c)[8]) {  // each column twice, as a pair
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            c[4 * m] = pack2(x.c[m].x, x.c[m].x);
            c[4 * m + 1] = pack2(x.c[m].y, x.c[m].y);
            c[4 * m + 2] = pack2(x.c[m].z, x.c[m].z);
            c[4 * m + 3] = pack2(x.c[m].w, x.c[m].w);
        }
    };
    // first row of the thread's pair i, first column of its run m of four columns
    auto row_of = [&](int i) { return (i >> 1) * (DKM / 2) + 4 * rg + 2 * (i & 1); };
    auto col_of = [&](int m) { return m * (kCols / 2) + 4 * cg; };

    f2 S[4][8];  // [pair of rows][column]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 8; ++c) S[i][c] = 0ull;

    if (nseg > 1) {
        // ---- the segment from zero: its end state and total decay.  A block of eight tokens at once,
        // S <- Diag(prod_j gamma_j) S + sum_j (k_j prod_{m > j} gamma_m)^T v_j: the suffix products
        // (all at most 1) are formed by the thread that stages a channel, which leaves one operation
        // per state element and token instead of two.
        f2 dec[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) dec[i] = pack2(1.f, 1.f);
        if (want_sum) {
            group_sync();
            int buf = 0;
            for (unsigned n = 0; n < nblk; ++n, buf ^= 1) {
                const float *st = sm + buf * Sh::stage;
                const Rows gg = rows_of(st + Sh::g, 0);
                Rows kn = rows_of(st + Sh::k, 0);
                Cols vn = cols_of(st + Sh::v, 0);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    dec[i] = mul2(dec[i], gg.r[i]);
#pragma unroll
                    for (int c = 0; c < 8; ++c) S[i][c] = mul2(gg.r[i], S[i][c]);
                }
#pragma unroll
                for (int j = 0; j < kTok; ++j) {  // (tokens past the segment: k = v = 0, gamma = 1)
                    const Rows kk = kn;
                    f2 vv[8];
                    spread(vn, vv);
                    if (j + 1 < kTok) {  // the next token's operands while this one's are used
                        kn = rows_of(st + Sh::k, j + 1);
                        vn = cols_of(st + Sh::v, j + 1);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int c = 0; c < 8; ++c) S[i][c] = fma2(kk.r[i], vv[c], S[i][c]);
                }
                group_sync();
            }
        }
        // the states of the CTA's groups become running ones, one group after the other: group grp's
        // is that of segments (first of the CTA) .. seg from zero, its decay their product
        for (int gi = 0; gi < G; ++gi) {
            if (grp == gi) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = row_of(i);
                    float2 d = unpack2(dec[i]);
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        const float2 x0 = unpack2(S[i][4 * m]), x1 = unpack2(S[i][4 * m + 1]);
                        const float2 x2 = unpack2(S[i][4 * m + 2]), x3 = unpack2(S[i][4 * m + 3]);
                        float4 lo = make_float4(x0.x, x1.x, x2.x, x3.x), hi = make_float4(x0.y, x1.y, x2.y, x3.y);
                        float *at = ss + r * kCols + col_of(m);
                        if (gi > 0) {
                            const float4 pl = *reinterpret_cast<const float4 *>(at - Sh::group);
                            const float4 ph = *reinterpret_cast<const float4 *>(at - Sh::group + kCols);
                            lo = make_float4(fmaf(d.x, pl.x, lo.x), fmaf(d.x, pl.y, lo.y), fmaf(d.x, pl.z, lo.z), fmaf(d.x, pl.w, lo.w));
                            hi = make_float4(fmaf(d.y, ph.x, hi.x), fmaf(d.y, ph.y, hi.y), fmaf(d.y, ph.z, hi.z), fmaf(d.y, ph.w, hi.w));
                        }
                        *reinterpret_cast<float4 *>(at) = lo;
                        *reinterpret_cast<float4 *>(at + kCols) = hi;
                    }
                    if (cg == 0) {
                        if (gi > 0) {
                            d.x *= sd[r - Sh::group];
                            d.y *= sd[r + 1 - Sh::group];
                        }
                        sd[r] = d.x;
                        sd[r + 1] = d.y;
                    }
                }
            }
            if (gi + 1 < G) __syncthreads();
        }
        cluster_arrive();
        cluster_wait();
        cluster_arrive();  // (the helpers read the peers' states before theirs)
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = row_of(i);
            const float2 d = grp > 0 ? make_float2(sd[r - Sh::group], sd[r + 1 - Sh::group]) : make_float2(1.f, 1.f);
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const float4 pl = *reinterpret_cast<const float4 *>(ps + r * kCols + col_of(m));
                const float4 ph = *reinterpret_cast<const float4 *>(ps + (r + 1) * kCols + col_of(m));
                float4 il = make_float4(0.f, 0.f, 0.f, 0.f), ih = il;
                if (grp > 0) {
                    il = *reinterpret_cast<const float4 *>(ss - Sh::group + r * kCols + col_of(m));
                    ih = *reinterpret_cast<const float4 *>(ss - Sh::group + (r + 1) * kCols + col_of(m));
                }
                S[i][4 * m] = pack2(fmaf(d.x, pl.x, il.x), fmaf(d.y, ph.x, ih.x));
                S[i][4 * m + 1] = pack2(fmaf(d.x, pl.y, il.y), fmaf(d.y, ph.y, ih.y));
                S[i][4 * m + 2] = pack2(fmaf(d.x, pl.z, il.z), fmaf(d.y, ph.z, ih.z));
                S[i][4 * m + 3] = pack2(fmaf(d.x, pl.w, il.w), fmaf(d.y, ph.w, ih.w));
            }
        }
        cluster_wait();
        __syncthreads();
    }
    if (t0 >= t1) return;
    group_sync();
    // ---- the tokens with their outputs.  Iteration n: the compute threads walk block n while the
    // helpers store block n - 1's outputs and stage block n + 1; one more iteration stores the last
    // block's.
    for (unsigned n = 0; n <= nblk; ++n) {
        const int buf = static_cast<int>(n & 1);
        if (n < nblk) {
            const float *st = sm + buf * Sh::stage;
            float *po = sm + Sh::po + buf * Sh::po_n;
            // column groups of odd row groups are stored 16 words away, so that a quarter warp's four
            // groups of two row groups fall into different banks
            const int pcol = 4 * (cg ^ ((rg & 1) << 2));
            Rows qn = rows_of(st + Sh::q, 0), kn = rows_of(st + Sh::k, 0), gn = rows_of(st + Sh::g, 0);
            Cols vn = cols_of(st + Sh::v, 0);
#pragma unroll
            for (int j = 0; j < kTok; ++j) {
                const Rows qq = qn, kk = kn, gg = gn;
                f2 vv[8], o[8];
                spread(vn, vv);
                if (j + 1 < kTok) {  // the next token's operands while this one's are used
                    qn = rows_of(st + Sh::q, j + 1);
                    kn = rows_of(st + Sh::k, j + 1);
                    gn = rows_of(st + Sh::g, j + 1);
                    vn = cols_of(st + Sh::v, j + 1);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        S[i][c] = fma2(gg.r[i], S[i][c], mul2(kk.r[i], vv[c]));
                        o[c] = i == 0 ? mul2(qq.r[i], S[i][c]) : fma2(qq.r[i], S[i][c], o[c]);
                    }
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const float2 a = unpack2(o[4 * m]), d = unpack2(o[4 * m + 1]);
                    const float2 e = unpack2(o[4 * m + 2]), f = unpack2(o[4 * m + 3]);
                    *reinterpret_cast<float4 *>(po + (j * RG + rg) * kCols + m * (kCols / 2) + pcol) =
                        make_float4(a.x + a.y, d.x + d.y, e.x + e.y, f.x + f.y);
                }
            }
        }
        group_sync();
    }
    if (p.final_state != nullptr && t1 == static_cast<unsigned>(T)) {
        float *fs = p.final_state + static_cast<long long>(bh) * Dk * Dv;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const int r = row_of(i), col = c0 + col_of(m);
                const float2 x0 = unpack2(S[i][4 * m]), x1 = unpack2(S[i][4 * m + 1]);
                const float2 x2 = unpack2(S[i][4 * m + 2]), x3 = unpack2(S[i][4 * m + 3]);
                float *lo = fs + static_cast<long long>(r) * Dv + col, *hi = lo + Dv;
                if constexpr (VEC) {  // (Dk and Dv are multiples of four: rows r and r + 1, columns as one)
                    if (col < Dv && r < Dk) {
                        *reinterpret_cast<float4 *>(lo) = make_float4(x0.x, x1.x, x2.x, x3.x);
                        *reinterpret_cast<float4 *>(hi) = make_float4(x0.y, x1.y, x2.y, x3.y);
                    }
                } else {
                    const float xl[4] = {x0.x, x1.x, x2.x, x3.x}, xh[4] = {x0.y, x1.y, x2.y, x3.y};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (col + e < Dv && r < Dk) lo[e] = xl[e];
                        if (col + e < Dv && r + 1 < Dk) hi[e] = xh[e];
                    }
                }
            }
    }
}

// Whole sequences in 16 value columns a CTA, for launches that would leave most of the tiles above empty
// (narrow_columns).  Thread (group, column) owns one column of S over the group's sixteenth of the Dk rows
// in registers; the readout is sixteen partial sums, added after every block of 16 tokens through shared
// memory.  Bound by the chain of tokens below about four CTAs an SM, above it by the issue of its
// broadcast shared-memory reads (three for two rows, against 96 packed operations a read in the tiles).
constexpr int kNarrowTok = 16, kNarrowCols = 16, kNarrowGroups = 16;

template <int DKM, typename E>
__global__ void __launch_bounds__(kSimtThreads) gla_simt_narrow_kernel(const __grid_constant__ SimtParams sp) {
    constexpr int RPT = DKM / kNarrowGroups;               // rows of S per thread
    constexpr int NQ = kNarrowTok * DKM / kSimtThreads;    // staged q / k / gamma values per thread
    static_assert(kNarrowTok * kNarrowCols == kSimtThreads, "one staged v value per thread");
    __shared__ __align__(16) float sq[kNarrowTok][DKM];
    __shared__ __align__(16) float sk[kNarrowTok][DKM];
    __shared__ __align__(16) float sgam[kNarrowTok][DKM];
    __shared__ float sv[kNarrowTok][kNarrowCols];
    __shared__ float po[kNarrowGroups][kNarrowTok][kNarrowCols];  // partial readouts of the block
    __shared__ int stok[kNarrowTok];

    const Problem &p = sp.p;
    const int bh = static_cast<int>(blockIdx.x), b = fdiv(bh, sp.fd_H), h = bh - b * p.H;
    const int c0 = static_cast<int>(blockIdx.y) * kNarrowCols;
    const int tid = static_cast<int>(threadIdx.x);
    const int cj = tid % kNarrowCols, grp = tid / kNarrowCols;  // column and row group owned
    const int Dk = p.Dk, Dv = p.Dv;
    const unsigned T = static_cast<unsigned>(p.T);
    const long long row0 = (static_cast<long long>(b) * p.T) * p.H + h;
    const E *q = static_cast<const E *>(p.q), *k = static_cast<const E *>(p.k);
    const E *v = static_cast<const E *>(p.v), *g = static_cast<const E *>(p.g);
    E *out = static_cast<E *>(p.out);

    // one block's inputs in registers (zeros / gamma = 1 past the sequence and past Dk, Dv:
    // padding contributes nothing)
    float rq[NQ], rk[NQ], rg[NQ], rv;
    int rt = 0;
    auto load_block = [&](unsigned s0) {
        const int n = static_cast<int>(T - s0 < kNarrowTok ? T - s0 : kNarrowTok);
#pragma unroll
        for (int m = 0; m < NQ; ++m) {
            const int idx = tid + m * kSimtThreads, j = idx / DKM, i = idx % DKM;
            float qv = 0.f, kv = 0.f, gam = 1.f;
            if (j < n && i < Dk) {
                const long long off = (row0 + static_cast<long long>(scan_token(sp, s0 + j)) * p.H) * Dk + i;
                qv = to_f32(q[off]);
                kv = to_f32(k[off]);
                gam = gamma_of(to_f32(g[off]));
            }
            rq[m] = qv;
            rk[m] = kv;
            rg[m] = gam;
        }
        const int j = tid / kNarrowCols, c = tid % kNarrowCols;
        rv = 0.f;
        if (j < n && c0 + c < Dv) rv = to_f32(v[(row0 + static_cast<long long>(scan_token(sp, s0 + j)) * p.H) * Dv + c0 + c]);
        rt = tid < n ? scan_token(sp, s0 + tid) : 0;
    };

    float S[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) S[i] = 0.f;

    load_block(0);
    for (unsigned s0 = 0; s0 < T; s0 += kNarrowTok) {
        const int n = static_cast<int>(T - s0 < kNarrowTok ? T - s0 : kNarrowTok);
        __syncthreads();  // the previous block's shared values and partials are consumed
#pragma unroll
        for (int m = 0; m < NQ; ++m) {
            const int idx = tid + m * kSimtThreads;
            sq[idx / DKM][idx % DKM] = rq[m];
            sk[idx / DKM][idx % DKM] = rk[m];
            sgam[idx / DKM][idx % DKM] = rg[m];
        }
        sv[tid / kNarrowCols][tid % kNarrowCols] = rv;
        if (tid < kNarrowTok) stok[tid] = rt;
        __syncthreads();
        if (s0 + kNarrowTok < T) load_block(s0 + kNarrowTok);  // in flight while this block runs
        for (int j = 0; j < n; ++j) {
            const float vj = sv[j][cj];
            float o0 = 0.f, o1 = 0.f;
#pragma unroll
            for (int i = 0; i < RPT; i += 2) {
                const int r = grp * RPT + i;
                S[i] = fmaf(sgam[j][r], S[i], sk[j][r] * vj);
                S[i + 1] = fmaf(sgam[j][r + 1], S[i + 1], sk[j][r + 1] * vj);
                o0 = fmaf(sq[j][r], S[i], o0);
                o1 = fmaf(sq[j][r + 1], S[i + 1], o1);
            }
            po[grp][j][cj] = o0 + o1;
        }
        __syncthreads();
        // the block's outputs: sum over the row groups, scattered to the spatial tokens
        const int j = tid / kNarrowCols, c = tid % kNarrowCols;
        if (j < n && c0 + c < Dv) {
            float o = 0.f;
#pragma unroll
            for (int r = 0; r < kNarrowGroups; ++r) o += po[r][j][c];
            out[(row0 + static_cast<long long>(stok[j]) * p.H) * Dv + c0 + c] = from_f32<E>(o);
        }
    }
    const int col = c0 + cj;
    if (p.final_state != nullptr && col < Dv) {
        float *fs = p.final_state + static_cast<long long>(bh) * Dk * Dv;
#pragma unroll
        for (int i = 0; i < RPT; ++i)
            if (grp * RPT + i < Dk) fs[static_cast<long long>(grp * RPT + i) * Dv + col] = S[i];
    }
}

// CTAs per sequence: a cluster of 2, 3, 4, 8 or 16 (at most max_cluster) whose groups take a segment
// each, or 0 for whole sequences, one per group.  The segments cost each token twice (the pass from zero is about half the
// work of the one with outputs), so they pay while the launch does not fill the SMs without them: two
// CTAs fit an SM, and the largest cluster that keeps all CTAs resident measured fastest (GB300, graph
// replays, Dk = Dv = 64, 1,600 tokens, us at cluster 0 / 2 / 3 / 4 / 8 / 16):
//     2 sequences  266 / 117 / 82 / 62 / 37 / 30      48 sequences  308 / 131 / 144 / 110 / 112 / 154
//    12 sequences  267 / 117 / 81 / 62 / 38 / 47      96 sequences  285 / 209 / 149 / 170 / 182 / 294
//    24 sequences  266 / 116 / 82 / 63 / 63 / 84     192 sequences  315 / 337 / 324 / 323 / 344 / 567
// Clusters of 6 and 12 were slower than 4 and 8 (they fill the GPCs badly), 16 pays only while one
// CTA an SM is enough.  A segment keeps at least two blocks of tokens.
int choose_cluster(const Problem &p, int n_sm, int groups, int max_cluster) {
    const long long units = static_cast<long long>(p.B) * p.H * ((p.Dv + kCols - 1) / kCols);
    const long long blocks = (p.T + kTok - 1) / kTok;
    for (const int c : {16, 8, 4, 3, 2})
        if (c <= max_cluster && units * c <= (c == kMaxCluster ? 1LL : 2LL) * n_sm && blocks >= 2LL * groups * c) return c;
    return 0;
}

// Whether a launch of whole sequences takes 16 value columns a CTA instead of tiles of 64.  The tiles walk
// a sequence of up to 32 key channels with one warp, compute all 64 columns however many there are, and
// take 1 to 2 us longer to start, so they lose (GB300, graph replays, us in tiles / in 16 columns):
//   Dk <= 32: up to 16 columns at any size (200 fp32 sequences of 1,600 tokens at 32 x 16 517 / 234, 2,000 of
//     256 240 / 151); wider ones up to five 16-column CTAs an SM, at 16 bits eight or, long, twelve (fp32 at
//     32 x 32: 400 of 256 tokens 75 / 69; fp16 608 of 1,600 954 / 660, but 350 of 256 at 32 x 64 91 / 107).
//   Dk <= 64: up to 16 columns (fp16 400 of 1,600 at 61 x 14 696 / 453, fp32 1,000 of 16 at 64 x 16 14.1 / 9.8), but
//     for long fp32 sequences of which the tiles keep one CTA an SM (200 of 1,600 280 / 368; 400 515 / 411);
//     up to 48 tokens in two CTAs an SM (24 of 32 at 64 x 64 8.7 / 5.8, 60 of 48 11.4 / 10.1; 152 of 32 8.8 / 10.8);
//     long 16-bit sequences of two column blocks in four (200 of 1,600 at 64 x 32 617 / 449, 350 717 / 870).
// Above 64 key channels the tiles win (200 of 256 at 128 x 16 78 / 95) but for one or two tokens (4.1 / 3.2).
bool narrow_columns(const Problem &p, int n_sm) {
    const long long ctas = static_cast<long long>(p.B) * p.H * ((p.Dv + kNarrowCols - 1) / kNarrowCols);
    const bool half = p.dtype != 0, one = p.Dv <= kNarrowCols;
    if (p.Dk > 64) return false;
    if (p.Dk <= 32) return one || ctas <= (half ? (p.T >= 1024 ? 12LL : 8LL) : 5LL) * n_sm;
    if (one) return half || p.T <= 256 || ctas > 2LL * n_sm;
    if (p.T <= 48) return ctas <= 2LL * n_sm;
    return half && p.T >= 1024 && p.Dv <= 2 * kNarrowCols && ctas <= 4LL * n_sm;
}

// Whether the current device can place a cluster of `cluster` CTAs of this kernel (one whose GPCs have
// few SMs, or a context limited to some of them, may not).  Asked once per device, kernel and size.
template <int DKM, typename E, bool VEC>
bool cluster_fits(int cluster, int dev) {
    static std::atomic<unsigned int> known[64] = {}, fits[64] = {};  // a bit per cluster size
    const unsigned int bit = 1u << cluster;
    if (dev >= 0 && dev < 64 && (known[dev].load(std::memory_order_acquire) & bit))
        return (fits[dev].load(std::memory_order_relaxed) & bit) != 0;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = static_cast<unsigned>(cluster);
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(cluster));
    cfg.blockDim = dim3(kSimtThreads);
    cfg.dynamicSmemBytes = SimtShape<DKM>::bytes;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gla_simt_kernel<DKM, E, VEC>, &cfg) != cudaSuccess) {
        n = 0;
        cudaGetLastError();  // a size the device does not take: the launch falls to a smaller one
    }
    if (dev >= 0 && dev < 64) {
        if (n > 0) fits[dev].fetch_or(bit, std::memory_order_relaxed);
        known[dev].fetch_or(bit, std::memory_order_release);
    }
    return n > 0;
}

template <int DKM, typename E>
cudaError_t launch_narrow(const SimtParams &sp, cudaStream_t stream) {
    const dim3 grid(static_cast<unsigned>(sp.n_seqs), static_cast<unsigned>((sp.p.Dv + kNarrowCols - 1) / kNarrowCols));
    gla_simt_narrow_kernel<DKM, E><<<grid, kSimtThreads, 0, stream>>>(sp);
    return cudaGetLastError();
}

template <int DKM, typename E, bool VEC>
cudaError_t launch_shape(const Problem &p, cudaStream_t stream) {
    using Sh = SimtShape<DKM>;
    static std::atomic<unsigned long long> set_on_devices(0);
    auto kernel = gla_simt_kernel<DKM, E, VEC>;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int n_sm = 0;
    if ((e = sm_count(&n_sm)) != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(set_on_devices.load(std::memory_order_relaxed) & bit)) {
        if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::bytes)) != cudaSuccess ||
            (e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
            return e;
        set_on_devices.fetch_or(bit);
    }
    SimtParams sp = {};
    sp.p = p;
    sp.fd_H = make_fastdiv(p.H);
    sp.fd_gh = make_fastdiv(p.grid_h);
    sp.n_seqs = p.B * p.H;
    int cluster = choose_cluster(p, n_sm, Sh::G, kMaxCluster);
    while (cluster > 0 && !cluster_fits<DKM, E, VEC>(cluster, dev)) cluster = choose_cluster(p, n_sm, Sh::G, cluster - 1);
    if constexpr (DKM <= 64) {
        if (cluster == 0 && narrow_columns(p, n_sm)) return launch_narrow<DKM, E>(sp, stream);
    }
    const long long blocks = (p.T + kTok - 1) / kTok;
    sp.nseg = cluster > 0 ? cluster * Sh::G : 1;
    sp.seg_len = (blocks + sp.nseg - 1) / sp.nseg * kTok;
    const long long ctas = cluster > 0 ? static_cast<long long>(sp.n_seqs) * cluster : (sp.n_seqs + Sh::G - 1LL) / Sh::G;
    const dim3 grid(static_cast<unsigned>(ctas), static_cast<unsigned>((p.Dv + kCols - 1) / kCols));
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = static_cast<unsigned>(cluster);
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kSimtThreads);
    cfg.dynamicSmemBytes = Sh::bytes;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = cluster > 1 ? 1 : 0;
    if ((e = cudaLaunchKernelEx(&cfg, kernel, sp)) != cudaSuccess) return e;
    return cudaGetLastError();
}

template <typename E, bool VEC>
cudaError_t launch_vec(const Problem &p, cudaStream_t stream) {
    if (p.Dk <= 32) return launch_shape<32, E, VEC>(p, stream);
    if (p.Dk <= 64) return launch_shape<64, E, VEC>(p, stream);
    return launch_shape<128, E, VEC>(p, stream);
}

template <typename E>
cudaError_t launch_typed(const Problem &p, cudaStream_t stream) {
    // rows of whole four-element vectors load and store as such
    return p.Dk % 4 == 0 && p.Dv % 4 == 0 ? launch_vec<E, true>(p, stream) : launch_vec<E, false>(p, stream);
}

// Output gate of Sec. 3.1 applied in place: one warp per (token, head) row of
// Dv <= 128 outputs; lane j takes columns j, j + 32, j + 64, j + 96.
template <typename E>
__global__ void __launch_bounds__(256) gate_epilogue_kernel(E *out, const E *r, const float *w, float eps,
                                                            long long rows, int Dv) {
    const long long row = static_cast<long long>(blockIdx.x) * 8 + (threadIdx.x >> 5);
    if (row >= rows) return;
    const int lane = threadIdx.x & 31;
    E *o_row = out + row * Dv;
    const E *r_row = r + row * Dv;
    float o[4];
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int col = lane + 32 * i;
        o[i] = col < Dv ? to_f32(o_row[col]) : 0.f;
        ss += o[i] * o[i];
    }
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, m);
    const float inv = rsqrtf(ss / static_cast<float>(Dv) + eps);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int col = lane + 32 * i;
        if (col < Dv) {
            const float z = to_f32(r_row[col]);
            const float silu = __fdividef(z, 1.f + __expf(-z));
            o_row[col] = from_f32<E>(silu * o[i] * inv * w[col]);
        }
    }
}

// The same gate for 16-byte vectors: LPR = Dv / VEC lanes per row, each moving
// VEC = 16 / sizeof(E) contiguous values (coalesced 16-byte loads and stores).  Memory-bound
// (r and o in, u out; part of o is still in L2).  A thread takes N vectors, 256 apart, with all
// of its loads issued before the first is used: with one vector each, 2048 threads an SM keep
// 64 KB of loads in flight for the length of their latency, then nothing while they reduce
// and store.  r is read once (streaming loads).  GB300, the mixer's time taken off: bf16
// 614400 rows of 64 (236 MB) 36.5 -> 32.4 us (N = 1 -> 4; 35.6 us at 2, 34.9 at 6).
template <typename E, int LPR, int N>
__global__ void __launch_bounds__(256) gate_epilogue_vec_kernel(E *out, const E *r, const float *w, float eps,
                                                                long long rows) {
    constexpr int VEC = 16 / static_cast<int>(sizeof(E));
    constexpr int Dv = LPR * VEC;
    const long long first = static_cast<long long>(blockIdx.x) * (256 * N) + threadIdx.x;
    const long long vecs = rows * LPR;
    const int part = static_cast<int>(threadIdx.x % LPR);
    uint4 ov[N], rv[N];
#pragma unroll
    for (int n = 0; n < N; ++n) {
        const long long gid = first + n * 256;
        rv[n] = gid < vecs ? __ldcs(reinterpret_cast<const uint4 *>(r) + gid) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int n = 0; n < N; ++n) {
        const long long gid = first + n * 256;
        ov[n] = gid < vecs ? reinterpret_cast<const uint4 *>(out)[gid] : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int n = 0; n < N; ++n) {
        const long long gid = first + n * 256;
        const E *oe = reinterpret_cast<const E *>(&ov[n]);
        const E *re = reinterpret_cast<const E *>(&rv[n]);
        float o[VEC];
        float ss = 0.f;
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            o[i] = to_f32(oe[i]);
            ss += o[i] * o[i];
        }
#pragma unroll
        for (int m = LPR / 2; m >= 1; m >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, m);
        const float inv = rsqrtf(ss / static_cast<float>(Dv) + eps);
        uint4 uv;
        E *ue = reinterpret_cast<E *>(&uv);
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            const float z = to_f32(re[i]);
            ue[i] = from_f32<E>(__fdividef(z, 1.f + __expf(-z)) * o[i] * inv * w[part * VEC + i]);
        }
        if (gid < vecs) reinterpret_cast<uint4 *>(out)[gid] = uv;
    }
}

template <typename E, int LPR>
cudaError_t launch_gate_vec(E *out, const E *r, const float *w, float eps, long long rows, cudaStream_t stream) {
    const long long blocks = (rows * LPR + 255) / 256;
    // four vectors a thread where one each is more than the SMs hold at once (8 blocks an SM);
    // below that every vector's thread is resident and a longer thread only adds latency
    int n_sm = 0;
    const cudaError_t e = sm_count(&n_sm);
    if (e != cudaSuccess) return e;
    const bool deep = blocks > 8LL * n_sm;
    const long long grid = deep ? (blocks + 3) / 4 : blocks;
    if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
    if (deep)
        gate_epilogue_vec_kernel<E, LPR, 4><<<static_cast<unsigned>(grid), 256, 0, stream>>>(out, r, w, eps, rows);
    else
        gate_epilogue_vec_kernel<E, LPR, 1><<<static_cast<unsigned>(grid), 256, 0, stream>>>(out, r, w, eps, rows);
    return cudaGetLastError();
}

template <typename E>
cudaError_t launch_gate_typed(const Problem &p, const Gate &gate, cudaStream_t stream) {
    const long long rows = static_cast<long long>(p.B) * p.T * p.H;
    E *out = static_cast<E *>(p.out);
    const E *r = static_cast<const E *>(gate.r);
    constexpr int VEC = 16 / static_cast<int>(sizeof(E));
    // rows of a 16-byte-multiple width take the vector kernel (row starts stay 16-byte aligned)
    switch (p.Dv % VEC == 0 ? p.Dv / VEC : 0) {
    case 1: return launch_gate_vec<E, 1>(out, r, gate.w, gate.eps, rows, stream);
    case 2: return launch_gate_vec<E, 2>(out, r, gate.w, gate.eps, rows, stream);
    case 4: return launch_gate_vec<E, 4>(out, r, gate.w, gate.eps, rows, stream);
    case 8: return launch_gate_vec<E, 8>(out, r, gate.w, gate.eps, rows, stream);
    case 16: return launch_gate_vec<E, 16>(out, r, gate.w, gate.eps, rows, stream);
    case 32: return launch_gate_vec<E, 32>(out, r, gate.w, gate.eps, rows, stream);
    default: break;
    }
    const long long blocks = (rows + 7) / 8;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    gate_epilogue_kernel<E><<<static_cast<unsigned>(blocks), 256, 0, stream>>>(out, r, gate.w, gate.eps, rows, p.Dv);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gate_epilogue(const Problem &p, const Gate &gate, cudaStream_t stream) {
    if (p.dtype == 0) return launch_gate_typed<float>(p, gate, stream);
    if (p.dtype == 1) return launch_gate_typed<__half>(p, gate, stream);
    return launch_gate_typed<__nv_bfloat16>(p, gate, stream);
}

SimtPlan simt_plan(const Problem &p, int n_sm, int max_cluster) {
    const int groups = p.Dk <= 32 ? SimtShape<32>::G : p.Dk <= 64 ? SimtShape<64>::G : SimtShape<128>::G;
    const int cluster = choose_cluster(p, n_sm, groups, max_cluster);
    return SimtPlan{cluster, cluster == 0 && narrow_columns(p, n_sm) ? kNarrowCols : kCols};
}

cudaError_t launch_simt(const Problem &p, cudaStream_t stream) {
    switch (p.dtype) {
    case 0: return launch_typed<float>(p, stream);
    case 1: return launch_typed<__half>(p, stream);
    default: return launch_typed<__nv_bfloat16>(p, stream);
    }
}

}  // namespace gtr
