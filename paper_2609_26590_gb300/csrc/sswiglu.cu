// sswiglu.cu -- Spatial SwiGLU between its two projections (Sec. 3.1, Eq.
// spatial_swiglu): Z = SiLU(X W_g) * DWConv3x3(X W_v) on the patch grid, the
// step the deployed S-SwiGLU kernel fuses (Sec. 4).
//
// Memory-bound: per token it reads F gate and F value elements and writes F
// outputs.  Work is cut into tiles of rows x columns of the grid (at most 40 columns)
// x one 128-byte channel slice (64 channels at 16 bits, 32 at fp32) of one image, one
// CTA per tile, two CTAs per SM, so that one CTA's TMA loads overlap the other's
// arithmetic.  A tile's value box covers one more row and column on every side: where
// it leaves the grid the tensor map returns zeros, which is exactly the convolution's
// zero padding; the gate box covers the tile's own tokens.  Neighbouring tiles re-read
// their halo, which L2 serves.
//
// A lane owns two channels (its 9 taps and bias as packed pairs in registers), a warp
// four columns, and it walks down the tile's rows with a 3 x 6 window of values in
// registers: per row six 4-byte (fp32: 8-byte) shared-memory reads of values and four
// of gates for eight outputs, accumulated with fma.rn.f32x2 (two IEEE fp32 operations
// per instruction, taps in the oracle's order), about 14 instructions an output.
// Measured on a GB300 (graph replays, identical bits) against one column and four
// channels a thread with scalar operations (about 26 instructions an output), which was
// bound by their issue: 32 x 40 x 40 x 1536 bf16 141 -> 93 us (5.1 TB/s, 74 % of the
// measured copy bandwidth), 8 x 80 x 80 x 2304 fp16 194 -> 133 us, one 40 x 40 x 768
// image 9.0 -> 4.7 us.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <atomic>
#include <cstdint>
#include <cstring>

#include "f32x2.cuh"
#include "fastdiv.cuh"
#include "gla_internal.h"
#include "tc_ptx.cuh"

namespace gtr {

__device__ unsigned int g_sswiglu_status;

namespace {

using namespace ptx;

constexpr int kSwMaxThreads = 320;
constexpr int kSwStageBudget = 108 * 1024;        // a tile's boxes (two CTAs per SM)
constexpr int kSwMaxRows = 32;
constexpr int kSwMaxCols = 40;                    // ten column groups, a warp (fp32: half a warp) each
constexpr uint64_t kSwWaitNs = 1000000000ull;     // 1 s: a tile's copies never take that long

struct SwParams {
    CUtensorMap vmap;       // value tensor: dims (F, W, Hg, B), box (slice, cols + 2, rows + 2, 1)
    CUtensorMap gmap;       // gate tensor: same dims, box (slice, cols, rows, 1)
    void *out;
    const float *weight;
    const float *bias;
    int grid_h, grid_w, F, rows, cols;
    FastDiv ntile_f, ntile_x, ntile_y;
    FastDiv ngroup;         // column groups of a tile: cols / 4
    int strip;              // rows a work item walks
    uint32_t vbytes, gbytes;  // bytes of the value box and of the gate box
};

// SiLU(z) = z / (1 + e^{-z}) of a pair, by the hardware's 2^x and 1/x.  Flushing their subnormal
// results changes nothing: 1 + e is 1 there, and z / (1 + e) is below 2^-120 where 1/(1 + e) is.
__device__ __forceinline__ f2 silu2(f2 z) {
    const float kNegLog2e = -1.4426950408889634f;
    const float2 t = unpack2(mul2(z, pack2(kNegLog2e, kNegLog2e)));
    float e0, e1, r0, r1;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(t.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(t.y));
    const float2 d = unpack2(add2(pack2(e0, e1), pack2(1.f, 1.f)));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(d.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(d.y));
    return mul2(z, pack2(r0, r1));
}

// A lane's two channels: `word` in memory, a packed fp32 pair in registers.
template <typename E> struct Pair;
template <> struct Pair<float> {
    using word = uint2;
    static __device__ __forceinline__ f2 load(word w) { return pack2(__uint_as_float(w.x), __uint_as_float(w.y)); }
    static __device__ __forceinline__ word store(f2 a) {
        const float2 x = unpack2(a);
        return make_uint2(__float_as_uint(x.x), __float_as_uint(x.y));
    }
};
template <> struct Pair<__half> {
    using word = uint32_t;
    static __device__ __forceinline__ f2 load(word w) {
        const float2 x = __half22float2(*reinterpret_cast<const __half2 *>(&w));
        return pack2(x.x, x.y);
    }
    static __device__ __forceinline__ word store(f2 a) {
        const float2 x = unpack2(a);
        const __half2 h = __floats2half2_rn(x.x, x.y);
        return *reinterpret_cast<const uint32_t *>(&h);
    }
};
template <> struct Pair<__nv_bfloat16> {
    using word = uint32_t;
    static __device__ __forceinline__ f2 load(word w) {
        return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
    }
    static __device__ __forceinline__ word store(f2 a) {
        const float2 x = unpack2(a);
        const __nv_bfloat162 h = __floats2bfloat162_rn(x.x, x.y);
        return *reinterpret_cast<const uint32_t *>(&h);
    }
};

template <typename E>
__global__ void __launch_bounds__(kSwMaxThreads, 2) sswiglu_kernel(const __grid_constant__ SwParams p) {
    using Word = typename Pair<E>::word;
    constexpr int LP = 128 / static_cast<int>(sizeof(Word));  // lanes per pixel: its 128-byte slice, two channels each
    constexpr int SLICE = 2 * LP;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    __shared__ uint64_t full;
    const int W = p.grid_w, TW = p.cols;
    // one tile per CTA (the grid has one CTA per tile): channel slice fastest, then columns, rows, image
    int rest = static_cast<int>(blockIdx.x);
    int nx = fdiv(rest, p.ntile_f);
    const int f0 = (rest - nx * p.ntile_f.d) * SLICE;
    rest = nx;
    nx = fdiv(rest, p.ntile_x);
    const int x0 = (rest - nx * p.ntile_x.d) * TW;
    const int b = fdiv(nx, p.ntile_y);
    const int y0 = (nx - b * p.ntile_y.d) * p.rows;
    if (threadIdx.x == 0) {
        mbar_init(&full, 1);
        fence_mbar_init();
        // the value box with its halo, then the gate box
        mbar_arrive_expect_tx(&full, p.vbytes + p.gbytes);
        tma_load_4d(smem, &p.vmap, &full, f0, x0 - 1, y0 - 1, b);
        tma_load_4d(smem + p.vbytes, &p.gmap, &full, f0, x0, y0, b);
    }
    __syncthreads();
    const int lane = static_cast<int>(threadIdx.x) % LP;
    const int fc = f0 + 2 * lane;
    const bool live = fc < p.F;
    f2 w[9], bs;
    {
        const float *w0 = p.weight + (size_t)(live ? fc : 0) * 9;
#pragma unroll
        for (int q = 0; q < 9; ++q) w[q] = pack2(w0[q], w0[9 + q]);
        bs = (live && p.bias != nullptr) ? pack2(p.bias[fc], p.bias[fc + 1]) : 0ull;
    }
    const bool ok = mbar_wait(&full, 0, nullptr, kSwWaitNs);
    if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) {  // never leave while the copies may still land
            atomicOr(&g_sswiglu_status, kStatusTimeout);
            mbar_wait(&full, 0, nullptr, kSwWaitNs);
        }
        __syncthreads();
        return;
    }
    const int R = p.grid_h - y0 < p.rows ? p.grid_h - y0 : p.rows;
    const int nstrip = (p.rows + p.strip - 1) / p.strip;
    const Word *vt = reinterpret_cast<const Word *>(smem) + lane;
    const Word *gt = reinterpret_cast<const Word *>(smem + p.vbytes) + lane;
    E *out = static_cast<E *>(p.out) + ((size_t)b * p.grid_h * W) * p.F + fc;
    // work items: four columns of the tile, walked down a strip of its rows with a 3 x 6 window of
    // values in registers (one new tile row of six per four outputs)
    for (int it = static_cast<int>(threadIdx.x) / LP; it < p.ngroup.d * nstrip; it += static_cast<int>(blockDim.x) / LP) {
        const int st = fdiv(it, p.ngroup), x = 4 * (it - st * p.ngroup.d);
        const int r0 = st * p.strip, r1 = r0 + p.strip < R ? r0 + p.strip : R;
        if (r0 >= r1 || x0 + x >= W || !live) continue;
        f2 win[3][6];
        const Word *vr = vt + ((size_t)r0 * (TW + 2) + x) * LP;
        auto load_row = [&](f2 (&row)[6]) {
#pragma unroll
            for (int j = 0; j < 6; ++j) row[j] = Pair<E>::load(vr[j * LP]);
            vr += (TW + 2) * LP;
        };
        load_row(win[0]);
        load_row(win[1]);
        const Word *gr = gt + ((size_t)r0 * TW + x) * LP;
        Word *dst = reinterpret_cast<Word *>(out + ((size_t)(y0 + r0) * W + x0 + x) * p.F);
        const int fw = p.F / 2, ncol = W - x0 - x;
        for (int r = r0; r < r1; r += 3) {
#pragma unroll
            for (int rr = 0; rr < 3; ++rr) {
                if (r + rr >= r1) break;
                // tile rows r + rr + {0, 1, 2} sit in window slots (rr + {0, 1, 2}) % 3
                load_row(win[(rr + 2) % 3]);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    f2 acc = bs;
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int j = 0; j < 3; ++j) acc = fma2(w[3 * i + j], win[(rr + i) % 3][c + j], acc);
                    const f2 z = mul2(silu2(Pair<E>::load(gr[c * LP])), acc);
                    if (c < ncol) dst[(size_t)c * fw] = Pair<E>::store(z);
                }
                gr += TW * LP;
                dst += (size_t)W * fw;
            }
        }
    }
}

int elem_bytes(int dtype) { return dtype == 0 ? 4 : 2; }

// Shared memory of a tile: the value box (rows + 2) x (cols + 2) and the gate box rows x cols,
// 128 bytes a token.
size_t stage_bytes(int rows, int cols) { return 128u * ((size_t)(rows + 2) * (cols + 2) + (size_t)rows * cols); }

// Columns and rows of a tile and the CTA's threads.  Large tiles re-read fewer halo rows (L2 serves
// them, but they cost the TMA unit the same): at 32 x 40 x 40 x 1536 in bf16 boxes of 36 / 54 / 72 /
// 108 KB ran in 154 / 114 / 103 / 93 us, so a tile takes as many rows as fit twice on an SM.  A launch
// that would not fill the SMs twice over with those takes the smallest tiles that still all run at
// once (one 40 x 40 image of 768 channels: 240 tiles 4.7 us, 120 tiles 4.9, 480 tiles 5.9; four of
// 20 x 20: 240 tiles 4.7 us, 336 tiles 6.1).
struct Tile {
    int rows, cols, strip, threads;
};
Tile choose_tile(const SwProblem &p, int n_sm) {
    Tile t;
    const int nx = (p.grid_w + kSwMaxCols - 1) / kSwMaxCols;
    t.cols = ((p.grid_w + nx - 1) / nx + 3) / 4 * 4;
    int r = 1;
    while (r < kSwMaxRows && r < p.grid_h && stage_bytes(r + 1, t.cols) <= kSwStageBudget) ++r;
    const int slice = 128 / elem_bytes(p.dtype);
    const long long per_row = (long long)p.B * ((p.grid_w + t.cols - 1) / t.cols) * ((p.F + slice - 1) / slice);
    auto tiles = [&](int rows) { return per_row * ((p.grid_h + rows - 1) / rows); };
    while (r > 1 && tiles(r - 1) <= 2LL * n_sm) --r;
    const int ny = (p.grid_h + r - 1) / r;
    t.rows = (p.grid_h + ny - 1) / ny;
    const int lp = p.dtype == 0 ? 16 : 32;
    const int groups = t.cols / 4;
    // as many warps as items, items split into strips of rows where columns alone are few
    int strips = 1;
    while (groups * strips * lp < 192 && strips < t.rows) ++strips;
    t.strip = (t.rows + strips - 1) / strips;
    strips = (t.rows + t.strip - 1) / t.strip;
    int th = groups * strips * lp;
    if (th > kSwMaxThreads) th = kSwMaxThreads;
    t.threads = (th + 31) / 32 * 32;
    return t;
}

template <typename E>
cudaError_t launch_typed(const SwParams &sp, unsigned grid, int threads, size_t smem, cudaStream_t stream) {
    static std::atomic<unsigned long long> set_on_devices(0);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(set_on_devices.load(std::memory_order_relaxed) & bit)) {
        e = cudaFuncSetAttribute(sswiglu_kernel<E>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSwStageBudget + 128);
        if (e != cudaSuccess) return e;
        set_on_devices.fetch_or(bit);
    }
    sswiglu_kernel<E><<<grid, threads, smem, stream>>>(sp);
    return cudaGetLastError();
}

bool encode(CUtensorMap *m, const SwProblem &p, const void *base, int box_w, int box_h) {
    auto enc = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(tensor_map_encoder());
    if (!enc) return false;
    const int es = elem_bytes(p.dtype);
    const cuuint64_t row = static_cast<cuuint64_t>(p.in_stride) * es;
    const cuuint64_t T = static_cast<cuuint64_t>(p.grid_h) * p.grid_w;
    cuuint64_t dims[4] = {static_cast<cuuint64_t>(p.F), static_cast<cuuint64_t>(p.grid_w),
                          static_cast<cuuint64_t>(p.grid_h), static_cast<cuuint64_t>(p.B)};
    cuuint64_t strides[3] = {row, row * p.grid_w, row * T};
    cuuint32_t box[4] = {static_cast<cuuint32_t>(128 / es), static_cast<cuuint32_t>(box_w),
                         static_cast<cuuint32_t>(box_h), 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUtensorMapDataType dt = p.dtype == 0 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : p.dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                                  : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    return enc(m, dt, 4, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool sswiglu_supported(const SwProblem &p) {
    // grids up to 254 columns: the entry point's documented range (the column tiles would take any width)
    return p.grid_w + 2 <= 256 && tensor_map_encoder() != nullptr;
}

cudaError_t launch_sswiglu(const SwProblem &p, cudaStream_t stream) {
    if (!sswiglu_supported(p)) return cudaErrorInvalidValue;
    const int slice = 128 / elem_bytes(p.dtype);
    int n_sm = 0;
    cudaError_t e = sm_count(&n_sm);
    if (e != cudaSuccess) return e;
    const Tile t = choose_tile(p, n_sm);
    SwParams sp;
    std::memset(&sp, 0, sizeof(sp));
    sp.rows = t.rows;
    sp.cols = t.cols;
    sp.strip = t.strip;
    sp.out = p.out;
    sp.weight = p.weight;
    sp.bias = p.bias;
    sp.grid_h = p.grid_h;
    sp.grid_w = p.grid_w;
    sp.F = p.F;
    sp.ntile_f = make_fastdiv((p.F + slice - 1) / slice);
    sp.ntile_x = make_fastdiv((p.grid_w + t.cols - 1) / t.cols);
    sp.ntile_y = make_fastdiv((p.grid_h + t.rows - 1) / t.rows);
    sp.ngroup = make_fastdiv(t.cols / 4);
    const long long tiles = (long long)p.B * sp.ntile_y.d * sp.ntile_x.d * sp.ntile_f.d;
    if (tiles <= 0 || tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    sp.vbytes = static_cast<uint32_t>(128u * (size_t)(t.rows + 2) * (t.cols + 2));
    sp.gbytes = static_cast<uint32_t>(128u * (size_t)t.rows * t.cols);
    if (!encode(&sp.vmap, p, p.value, t.cols + 2, t.rows + 2) || !encode(&sp.gmap, p, p.gate, t.cols, t.rows))
        return cudaErrorInvalidValue;
    const unsigned grid = static_cast<unsigned>(tiles);  // one CTA per tile
    const size_t smem = (size_t)sp.vbytes + sp.gbytes + 128;
    if (p.dtype == 0) return launch_typed<float>(sp, grid, t.threads, smem, stream);
    if (p.dtype == 1) return launch_typed<__half>(sp, grid, t.threads, smem, stream);
    return launch_typed<__nv_bfloat16>(sp, grid, t.threads, smem, stream);
}

cudaError_t read_and_clear_sswiglu_status(unsigned int *status) {
    cudaError_t e = cudaMemcpyFromSymbol(status, g_sswiglu_status, sizeof(unsigned int));
    if (e != cudaSuccess) return e;
    const unsigned int zero = 0;
    return cudaMemcpyToSymbol(g_sswiglu_status, &zero, sizeof(unsigned int));
}

}  // namespace gtr
