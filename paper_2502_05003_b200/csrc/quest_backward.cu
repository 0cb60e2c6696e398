// QuEST training backward for one linear layer (Algorithm 2) on sm_100a:
//
//   dL/dxq_h = dL/dy wq_h                      dL/dx = IHT(M(x_h; xq_h) * dL/dxq_h)
//   dL/dwq_h = dL/dy^T xq_h                    dL/dw = IHT(M(w_h; wq_h) * dL/dwq_h)
//
// The products run in 16-bit precision on the tensor cores (Section 3.3, "Implementation").  dL/dy is
// used as it is (bfloat16); the quantized operand is dequantised to bfloat16, xq_h = bf16(sx[m] c_x),
// wq_h = bf16(sw[n] c_w) with c = 2k - (2^b - 1): one rounding per product.  Nothing is transposed: the
// tensor cores read an operand whose memory rows run along the contraction index as an MN-major
// operand (quest_gemm.cu).  Stages:
//   1. dequant_codes_kernel   wq_h [N x K], xq_h [M x K] from the packed codes and scales
//   2. gemm (bfloat16 mode)   d1[m][k] = M_x[m][k] sum_n dy[m][n] wq_h[n][k]   (dy K-major, wq_h MN-major)
//                             d2[n][k] = M_w[n][k] sum_m dy[m][n] xq_h[m][k]   (dy and xq_h MN-major)
//   3. iht_wide / iht_rows    block Hadamard transform, 1/sqrt(g), store in the output type
//      (for blocks of up to 128 stages 2 and 3 are one kernel: the transform runs in the GEMM epilogue,
//      where a thread holds 128 aligned columns of its output row)
//   A product whose output is small and whose sum is long runs in parts of the contraction index, or it would leave most
//   SMs idle; then stage 3 adds the parts (in order) and applies the mask, at any block size.
#include <cuda_bf16.h>
#include <math.h>

#include "quest_internal.cuh"

namespace quest {
namespace {

__device__ __forceinline__ uint16_t bf16_bits(float v) {
    __nv_bfloat16 h = __float2bfloat16_rn(v);
    return *reinterpret_cast<uint16_t *>(&h);
}

// Packed level indices and per-row scales -> dequantised values bf16(scale[r] * c) [rows x K], dense, up to two
// tensors per launch (CTAs from blocks0 on work on the second).  A CTA converts `rpb` whole rows, or (SPLIT)
// `piece` units of one row, gridDim.y of them: a few long rows would leave most SMs without a CTA.  A unit is sixteen
// consecutive elements (one 32-byte store; K % 32 == 0 keeps them in one row); two per thread and step are in flight.  Bound by
// the writes (2 B/element) once the arithmetic is out of the way: the row of a unit comes from a multiplication
// (`magic` = ceil(2^32 / units), exact below 2^20 units per CTA) instead of a 64-bit division, and 2k - (2^b - 1) from
// a packed multiply-add on 2^22 + k (the level in the low bits) instead of integer conversions, both exact.
// 4096 x 2048 + 2048 x 2048 elements at four bits: 10.4 -> 6.9 us.
struct DequantTensor {
    const uint8_t *codes;
    const float *scales;
    uint16_t *out;
    long long rows;
};
template <int CB, bool SPLIT>
__global__ void __launch_bounds__(256)
dequant_codes_kernel(DequantTensor t0, DequantTensor t1, int blocks0, int rpb, int piece, int units, uint32_t magic, int bits) {
    pdl_launch_dependents();
    pdl_wait();
    const bool second = (int)blockIdx.x >= blocks0;
    const DequantTensor t = second ? t1 : t0;
    const long long row0 = (long long)(second ? (int)blockIdx.x - blocks0 : (int)blockIdx.x) * rpb;
    const int rows_here = t.rows - row0 < rpb ? (int)(t.rows - row0) : rpb;
    const int begin = SPLIT ? (int)blockIdx.y * piece : 0;
    const int n = SPLIT ? min(units - begin, piece) : rows_here * units;
    const long long first = row0 * units + begin;            // the CTA's first unit
    const uint32_t *c32 = reinterpret_cast<const uint32_t *>(t.codes);
    const float off = -(8388608.0f + (float)((1 << bits) - 1));
    const float2 two = make_float2(2.0f, 2.0f), off2 = make_float2(off, off);
    constexpr int NW = CB >= 2 ? CB / 2 : 1;                 // words that hold the levels of a unit
    for (int i0 = threadIdx.x; i0 < n; i0 += 2 * 256) {
        float sc[2];
        uint32_t lv[2][NW];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = i0 + 256 * u;
            if (i < n) {
                const long long o = first + i;
                sc[u] = __ldg(t.scales + row0 + __umulhi((uint32_t)i, magic));
                if constexpr (CB == 1) {
                    lv[u][0] = (__ldg(c32 + (o >> 1)) >> (16 * (int)(o & 1))) & 0xFFFFu;
                } else {
#pragma unroll
                    for (int q = 0; q < NW; ++q) lv[u][q] = __ldg(c32 + NW * o + q);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = i0 + 256 * u;
            if (i >= n) break;
            const float2 sc2 = make_float2(sc[u], sc[u]);
            uint32_t r[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t w = lv[u][(2 * j * CB) / 32];
                const int s0 = (2 * j * CB) % 32;
                const uint32_t mask = ((1u << CB) - 1u) << 1;    // the level one bit up: 2^22 + k
                const float2 k = make_float2(__uint_as_float(((s0 ? w >> (s0 - 1) : w << 1) & mask) | 0x4A800000u),
                                             __uint_as_float(((w >> (s0 + CB - 1)) & mask) | 0x4A800000u));
                const float2 v = __fmul2_rn(sc2, __ffma2_rn(k, two, off2));
                const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
                r[j] = *reinterpret_cast<const uint32_t *>(&h);
            }
            store32B(t.out + (first + i) * 16, r);
        }
    }
}

// Inverse orthonormal block Hadamard transform of every row of d [rows x cols] (binary32, dense),
// stored as out_dtype, dense.  Every thread owns 32 contiguous elements; descending
// stride: partners in other warps through shared memory, partners in this warp through shuffles,
// the rest in registers.  A row of T = cols/32 threads occupies S slots as in the quantizer.
// PARTS: d is `parts` matrices `part_stride` elements apart, whose sum, where `mask` [rows x cols/8] keeps it, is the input
// (blocks of up to 1024: see transform_adds_parts).
template <bool PARTS>
__global__ void __launch_bounds__(512)
iht_rows_kernel(const float *__restrict__ d, long long rows, int cols, int had_block, float inv_sqrt_g, void *__restrict__ out,
                int out_dtype, int S, int R, int parts, long long part_stride, const uint8_t *__restrict__ mask) {
    extern __shared__ float xsm[];                 // [32][blockDim.x] exchange
    pdl_launch_dependents();
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31, nthreads = blockDim.x;
    const int r_local = tid / S;
    const int tr = tid - r_local * S;
    const long long row = (long long)blockIdx.x * R + r_local;
    const bool active = row < rows && tr < cols / 32;
    float v[32];
    if (active) {
        // d is in the workspace (256-byte aligned), rows are multiples of 128 bytes
        const float *src = d + row * cols + (long long)tr * 32;
        uint32_t w[32];
#pragma unroll
        for (int q = 0; q < 4; ++q) load32B(src + 8 * q, &w[8 * q]);
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(w[i]);
        if constexpr (PARTS) {
            const uint32_t keep = __ldg(reinterpret_cast<const uint32_t *>(mask + row * (cols >> 3)) + tr);
#pragma unroll 2
            for (int q2 = 1; q2 < parts; ++q2) {
                src += part_stride;
#pragma unroll
                for (int q = 0; q < 4; ++q) load32B(src + 8 * q, &w[8 * q]);
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] += __uint_as_float(w[i]);
            }
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = (keep >> i) & 1u ? v[i] : 0.0f;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = 0.0f;
    }
    if constexpr (!PARTS) {
        for (int s = had_block >> 1; s >= 1024; s >>= 1) {     // partner thread is in another warp
            const int dist = s >> 5;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 32; ++i) xsm[i * nthreads + tid] = v[i];
            __syncthreads();
            const float sg = (tid & dist) ? -1.0f : 1.0f;
            const int pt = tid ^ dist;
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = fmaf(v[i], sg, xsm[i * nthreads + pt]);
        }
    }
    {
        int s0 = had_block >> 1;
        if (s0 > 512) s0 = 512;
#pragma unroll 1
        for (int s = s0; s >= 32; s >>= 1) {                   // partner thread is a lane of this warp
            const int dist = s >> 5;
            const float sg = (lane & dist) ? -1.0f : 1.0f;
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = fmaf(v[i], sg, __shfl_xor_sync(0xffffffffu, v[i], dist));
        }
    }
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        if (s < had_block) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if ((i & s) == 0) {
                    const float a = v[i], b = v[i + s];
                    v[i] = a + b;
                    v[i + s] = a - b;
                }
        }
    }
    if (!active) return;
    if (out_dtype == QUEST_F32) {
        uint32_t w[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) w[i] = __float_as_uint(v[i] * inv_sqrt_g);
        store_words(reinterpret_cast<float *>(out) + row * cols + (long long)tr * 32, w);
    } else {
        uint32_t w[16];
#pragma unroll
        for (int i = 0; i < 16; ++i)
            w[i] = (uint32_t)bf16_bits(v[2 * i] * inv_sqrt_g) | ((uint32_t)bf16_bits(v[2 * i + 1] * inv_sqrt_g) << 16);
        store_words(reinterpret_cast<uint16_t *>(out) + row * cols + (long long)tr * 32, w);
    }
}

// The same transform for blocks of g = 2^L = 256 .. 4096, 64 elements per thread.  Phase A: the g/64 threads of a
// block take pairs of neighbouring elements 2p + 64 j apart (2p + 128 j at g = 4096), so that the strides g/2 .. 64
// (.. 128) stay in a thread's registers and a warp reads consecutive memory.  The result goes through shared memory
// in row order (16 bytes of padding per 64 elements: no bank conflicts either way); phase B takes 64 contiguous
// elements (at g = 4096 first stride 64 against the neighbouring thread's), strides 32 .. 1, and the scaled output
// goes back through the same shared memory so that it leaves in consecutive 16-byte stores.  The order of the stages
// and every operand are those of the kernel above: identical results.
// Bound by memory traffic (the masked product is read from L2, where the contraction left it).
template <int L, bool PARTS>
__global__ void __launch_bounds__(128, 4)
iht_wide_kernel(const float *__restrict__ d, long long rows, int cols, float inv_sqrt_g, void *__restrict__ out,
                int out_dtype, int S, int R, int parts, long long part_stride, const uint8_t *__restrict__ mask) {
    extern __shared__ __align__(16) float tbuf[];              // [R][cols + cols / 16]
    constexpr int NA = L == 12 ? 5 : L - 6;                    // strides of phase A
    constexpr int NL = 5 - NA;
    constexpr int HI = L == 12 ? 128 : 64;                     // elements between the pairs that phase A combines
    constexpr int TB = 1 << (L - 6);                           // threads per rotation block
    pdl_launch_dependents();
    pdl_wait();
    const int tid = threadIdx.x;
    const int r_local = tid / S;
    const int tr = tid - r_local * S;
    const long long row0 = (long long)blockIdx.x * R;
    const long long row = row0 + r_local;
    const bool active = row < rows && tr < (cols >> 6);
    const int pitch = cols + (cols >> 4);
    float *trow = tbuf + (size_t)r_local * pitch;
    float2 v[32];
    const float2 neg1 = make_float2(-1.0f, -1.0f);
    if (active) {
        const int p = tr & (TB - 1);
        const int i0 = (tr / TB) * (1 << L) + 2 * p;           // first element of this thread's pairs
        const float *src = d + row * cols + i0;
#pragma unroll
        for (int j = 0; j < 32; ++j)
            v[j] = __ldg(reinterpret_cast<const float2 *>(src + (j >> NL) * HI + 2 * ((j & ((1 << NL) - 1)) << NA)));
        if constexpr (PARTS) {
            for (int q = 1; q < parts; ++q) {
                src += part_stride;
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    v[j] = __fadd2_rn(v[j], __ldg(reinterpret_cast<const float2 *>(src + (j >> NL) * HI + 2 * ((j & ((1 << NL) - 1)) << NA))));
            }
            const uint8_t *mrow = mask + row * (cols >> 3);
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const int e = i0 + (j >> NL) * HI + 2 * ((j & ((1 << NL) - 1)) << NA);
                const uint32_t keep = (uint32_t)__ldg(mrow + (e >> 3)) >> (e & 7);
                v[j] = make_float2(keep & 1u ? v[j].x : 0.0f, keep & 2u ? v[j].y : 0.0f);
            }
        }
#pragma unroll
        for (int s = 16; s >= (1 << NL); s >>= 1)
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if ((j & s) == 0) {
                    const float2 a = v[j], b = v[j + s];
                    v[j] = __fadd2_rn(a, b);
                    v[j + s] = __ffma2_rn(b, neg1, a);
                }
        float *dst = trow + i0 + ((i0 >> 6) << 2);
#pragma unroll
        for (int j = 0; j < 32; ++j)
            *reinterpret_cast<float2 *>(dst + (j >> NL) * (HI + HI / 16) + 2 * ((j & ((1 << NL) - 1)) << NA)) = v[j];
    }
    __syncthreads();
    if (active) {
        const float4 *own = reinterpret_cast<const float4 *>(trow + tr * 68);
        if constexpr (L == 12) {
            const float4 *oth = reinterpret_cast<const float4 *>(trow + (tr ^ 1) * 68);
            const float sg = (tr & 1) ? -1.0f : 1.0f;
            const float2 sg2 = make_float2(sg, sg);
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const float4 a = own[q], b = oth[q];
                v[2 * q] = __ffma2_rn(make_float2(a.x, a.y), sg2, make_float2(b.x, b.y));
                v[2 * q + 1] = __ffma2_rn(make_float2(a.z, a.w), sg2, make_float2(b.z, b.w));
            }
        } else {
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const float4 a = own[q];
                v[2 * q] = make_float2(a.x, a.y);
                v[2 * q + 1] = make_float2(a.z, a.w);
            }
        }
#pragma unroll
        for (int s = 16; s >= 1; s >>= 1)
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if ((j & s) == 0) {
                    const float2 a = v[j], b = v[j + s];
                    v[j] = __fadd2_rn(a, b);
                    v[j + s] = __ffma2_rn(b, neg1, a);
                }
        const float2 sc = make_float2(inv_sqrt_g, inv_sqrt_g);
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = __fmul2_rn(make_float2(v[j].x + v[j].y, v[j].x - v[j].y), sc);
    }
    if constexpr (L == 12) __syncthreads();                    // the neighbour has read this thread's elements
    if (active) {
        if (out_dtype == QUEST_F32) {
            float4 *o = reinterpret_cast<float4 *>(trow + tr * 68);
#pragma unroll
            for (int q = 0; q < 16; ++q) o[q] = make_float4(v[2 * q].x, v[2 * q].y, v[2 * q + 1].x, v[2 * q + 1].y);
        } else {
            uint4 *o = reinterpret_cast<uint4 *>(trow + tr * 68);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                uint32_t w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const __nv_bfloat162 h = __floats2bfloat162_rn(v[4 * q + j].x, v[4 * q + j].y);
                    w[j] = *reinterpret_cast<const uint32_t *>(&h);
                }
                o[q] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    }
    __syncthreads();
    // coalesced stores: 16-byte chunk c of a row belongs to thread c / 16 (binary32) or c / 8 (bfloat16) of the row
    const int sh = out_dtype == QUEST_F32 ? 4 : 3;
    const int chunks = cols >> (6 - sh);
    const long long left = rows - row0;
    const int rows_here = left < R ? (int)left : R;
    const size_t row_bytes = (size_t)cols * (out_dtype == QUEST_F32 ? 4 : 2);
    for (int r = 0; r < rows_here; ++r) {
        uint4 *dst = reinterpret_cast<uint4 *>(reinterpret_cast<uint8_t *>(out) + (size_t)(row0 + r) * row_bytes);
        const float *from = tbuf + (size_t)r * pitch;
        for (int c = tid; c < chunks; c += (int)blockDim.x)
            dst[c] = *reinterpret_cast<const uint4 *>(from + (c >> sh) * 68 + (c & ((1 << sh) - 1)) * 4);
    }
}

struct BwdWorkspace {
    uint16_t *wh, *xh;      // dequantised operands [N x K], [M x K]
    float *d1, *d2;         // masked products when the inverse transform is a separate kernel
    size_t bytes;
};
BwdWorkspace carve_bwd(void *base, int64_t M, int64_t N, int64_t K) {
    BwdWorkspace w;
    uint8_t *b = reinterpret_cast<uint8_t *>(base);
    size_t off = 0;
    auto take = [&](size_t n) { uint8_t *p = b + off; off += align_up(n, 256); return p; };
    w.wh = reinterpret_cast<uint16_t *>(take((size_t)N * K * 2));
    w.xh = reinterpret_cast<uint16_t *>(take((size_t)M * K * 2));
    w.d1 = reinterpret_cast<float *>(take((size_t)M * K * 4));
    w.d2 = reinterpret_cast<float *>(take((size_t)N * K * 4));
    w.bytes = off;
    return w;
}

// Rows per CTA of a transform whose rows take S threads: CTAs of 128 threads where a row fits.  Adding parts is bound by the
// reads in flight, so there the rows are dealt out until every SM has several CTAs.
int transform_rows_per_cta(int64_t rows, int S, int parts) {
    int R = S <= 128 ? 128 / S : 1;
    while (parts > 1 && R > 1 && R * S > 32 && rows < 4ll * num_sms() * R) R >>= 1;
    return R;
}

// A transform launched ahead of its predecessor's end, or (adding parts, and where its launcher says so) plainly.
template <typename... KArgs, typename... Args>
cudaError_t launch_transform(void (*kernel)(KArgs...), int64_t grid, int threads, size_t smem, cudaStream_t st, bool ahead, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = ahead ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

template <int L>
cudaError_t launch_iht_wide(const float *d, int64_t rows, int64_t cols, int had_block, void *out, int out_dtype, int parts,
                            const uint8_t *mask, cudaStream_t st) {
    const int T = (int)(cols >> 6);                            // at most 128 (cols <= 8192)
    int S = 1;
    while (S < T) S <<= 1;
    const int R = transform_rows_per_cta(rows, S, parts);
    const size_t smem = sizeof(float) * (size_t)R * (size_t)(cols + cols / 16);      // at most 34 KB
    // Launched ahead, the CTAs settle on the few SMs that the gradient product leaves free and run there several to an SM
    // while the others idle: an input gradient of 0.3 to 5 Mi elements launched plainly takes 0.72 .. 0.93 of the time
    // (204 shapes, at most 1.02).  A grid of a few waves levels that and gains the launch, 0.96 from 6 Mi elements on, and so
    // does one that fits those SMs.
    const int64_t elements = rows * cols;
    const bool ahead = parts == 1 && (elements < (300 << 10) || elements >= (5 << 20));
    return launch_transform(parts > 1 ? iht_wide_kernel<L, true> : iht_wide_kernel<L, false>, (rows + R - 1) / R, R * S, smem, st, ahead, d,
                            (long long)rows, (int)cols, 1.0f / sqrtf((float)had_block), out, out_dtype, S, R, parts,
                            (long long)((rows + 255) / 256 * 256 * cols), mask);
}

// Any block size, one thread per 32 elements.
int launch_iht_rows(const float *d, int64_t rows, int64_t cols, int had_block, void *out, int out_dtype, int parts,
                    const uint8_t *mask, cudaStream_t st) {
    const int T = (int)(cols / 32);
    int S;
    if (T < 32) { S = 1; while (S < T) S <<= 1; } else { S = (T + 31) / 32 * 32; }
    const int R = transform_rows_per_cta(rows, S, parts);
    const int threads = R * S;
    const size_t smem = had_block >= 2048 ? sizeof(float) * 32 * (size_t)threads : 0;
    if (smem > 48 * 1024) {
        static DynamicSmemOnce once;
        const cudaError_t e = once.set(iht_rows_kernel<false>, 72 * 1024);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    // Launched ahead, the CTAs gather on the SMs that the gradient product leaves free, as in launch_iht_wide; eight of them
    // fit on an SM.  Plainly an output of 0.5 to 0.9 Mi elements takes 0.4 .. 0.8 us less, of 1 to 3 Mi 1.2 .. 2.1 us less,
    // below 0.3 and above 4 Mi elements up to 0.6 us more (300 backward passes).
    const int64_t elements = rows * cols;
    const bool ahead = parts == 1 && (elements < (400 << 10) || elements >= (4 << 20));
    const cudaError_t e = launch_transform(parts > 1 ? iht_rows_kernel<true> : iht_rows_kernel<false>, (rows + R - 1) / R, threads, smem, st,
                                           ahead, d, (long long)rows, (int)cols, had_block, 1.0f / sqrtf((float)had_block), out,
                                           out_dtype, S, R, parts, (long long)((rows + 255) / 256 * 256 * cols), mask);
    return e == cudaSuccess ? QUEST_OK : cuda_fail(e);
}

// Whether a transform that adds parts serves these rows.  It has no exchange between warps for the general kernel, which
// blocks of 8192 and more take, and blocks of 2048 and 4096 in rows above 8192 columns; their 64 column tiles and more
// leave 74 pairs nothing to divide among anyway.
bool transform_adds_parts(int64_t cols, int had_block) { return had_block <= 1024 || (had_block <= 4096 && cols <= 8192); }

// Inverse transform of d [rows x cols], binary32 and dense, or (parts > 1) of the sum of the parts that
// launch_gemm_bf16_parts left there, where `mask` keeps it; `out` is dense too.
int launch_iht(const float *d, int64_t rows, int64_t cols, int had_block, void *out, int out_dtype, int parts,
               const uint8_t *mask, cudaStream_t st) {
    // blocks of 256 .. 4096 in rows that one CTA holds with 64 elements per thread.  Small outputs of narrow blocks stay
    // with the general kernel: its CTAs are many and short, and the fewer strides leave a thread the less there is to gain.
    // General kernel's time over this one's, contraction and dequantisation included: g = 256 0.7 .. 0.95 below
    // 9/16 Mi elements, 1.0 at 0.75, 1.1 at 1.5, 1.15 from 4 Mi on, but 0.75 .. 0.85 up to 2 Mi in rows of one block;
    // g = 512 0.8 .. 0.95 up to half a Mi, 1.05 at 0.75 .. 2, 1.2 from 4 on; g = 1024 0.8 .. 1.0 up to a quarter Mi
    const int64_t few = cols == 256 ? 4 << 20 : cols > 4096 ? 0 : had_block <= 512 ? 9 << 16 : had_block == 1024 ? 5 << 16 : 0;
    if (rows * cols >= few && had_block >= 256 && had_block <= 4096 && cols <= 8192) {
        cudaError_t e;
        switch (had_block) {
            case 256: e = launch_iht_wide<8>(d, rows, cols, had_block, out, out_dtype, parts, mask, st); break;
            case 512: e = launch_iht_wide<9>(d, rows, cols, had_block, out, out_dtype, parts, mask, st); break;
            case 1024: e = launch_iht_wide<10>(d, rows, cols, had_block, out, out_dtype, parts, mask, st); break;
            case 2048: e = launch_iht_wide<11>(d, rows, cols, had_block, out, out_dtype, parts, mask, st); break;
            default: e = launch_iht_wide<12>(d, rows, cols, had_block, out, out_dtype, parts, mask, st); break;
        }
        return e == cudaSuccess ? QUEST_OK : cuda_fail(e);
    }
    return launch_iht_rows(d, rows, cols, had_block, out, out_dtype, parts, mask, st);
}

bool bwd_shape_ok(int64_t M, int64_t N, int64_t K) {
    return M > 0 && N > 0 && K >= 32 && K % 32 == 0 && K <= 16384 && M % 8 == 0 && N % 8 == 0 &&
           M <= ((int64_t)1 << 24) && N <= ((int64_t)1 << 24);
}

}  // namespace
}  // namespace quest

using namespace quest;

extern "C" size_t quest_bwd_workspace_bytes(int64_t M, int64_t N, int64_t K) {
    if (!bwd_shape_ok(M, N, K)) return 0;
    return carve_bwd(nullptr, M, N, K).bytes;
}

extern "C" int quest_linear_bwd(const void *dy, int64_t M, int64_t N, int64_t K, int bits, int had_block,
                                const uint8_t *xq, const float *sx, const uint8_t *mx,
                                const uint8_t *wq, const float *sw, const uint8_t *mw,
                                void *dx, void *dw, int out_dtype,
                                void *workspace, size_t workspace_bytes, void *stream) {
    if (!dy || !xq || !sx || !mx || !wq || !sw || !mw) return QUEST_ERR_NULL;
    if (!dx && !dw) return QUEST_ERR_NULL;
    if (bits < 1 || bits > 8) return QUEST_ERR_BITS;
    if (!bwd_shape_ok(M, N, K)) return QUEST_ERR_SHAPE;
    if (had_block < 1 || (had_block & (had_block - 1)) != 0 || had_block > K || K % had_block != 0)
        return QUEST_ERR_HAD_BLOCK;
    if (out_dtype != QUEST_F32 && out_dtype != QUEST_BF16) return QUEST_ERR_DTYPE;
    auto al = [](const void *p, size_t a) { return reinterpret_cast<uintptr_t>(p) % a == 0; };
    if (!al(dy, 16) || !al(mx, 16) || !al(mw, 16) || !al(sw, 4) || !al(sx, 4) || !al(xq, 4) || !al(wq, 4) || (dx && !al(dx, 16)) ||
        (dw && !al(dw, 16)))
        return QUEST_ERR_ALIGN;
    if (!workspace || !al(workspace, 256) || workspace_bytes < quest_bwd_workspace_bytes(M, N, K))
        return QUEST_ERR_WORKSPACE;
    int s = check_device();
    if (s) return s;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    BwdWorkspace ws = carve_bwd(workspace, M, N, K);
    struct Stage {                                   // RAII bracket for quest_stage_timing
        void *h;
        Stage(int id, cudaStream_t s_) : h(stage_begin(id, s_)) {}
        ~Stage() { stage_end(h); }
    };
    {
        // both dequantised operands in one launch, then the two products back to back
        Stage prep(QUEST_STAGE_UNPACK, st);
        const DequantTensor tw = {wq, sw, ws.wh, dx ? (long long)N : 0}, tx = {xq, sx, ws.xh, dw ? (long long)M : 0};
        const int units = (int)(K / 16);                     // at most 1024
        // about two units per thread, fewer while that would leave an SM less than about eight CTAs (7016 x 512 + 768 x 512
        // elements: 1.1 us slower with two than with fewer)
        int per_cta = 512;
        while (per_cta > 128 && (tw.rows + tx.rows) * units < 1184ll * per_cta) per_cta >>= 1;
        const int rpb = (per_cta + units - 1) / units;
        const int blocks0 = (int)((tw.rows + rpb - 1) / rpb);
        const int blocks = blocks0 + (int)((tx.rows + rpb - 1) / rpb);
        // rows shared by several CTAs only where there are fewer rows than two per SM (64 x 8192: 0.7 us; 1536 x 5504 would
        // take 2.9 us longer)
        const int parts = rpb == 1 && blocks < 2 * num_sms() ? (units + 127) / 128 : 1;
        const int piece = (units + parts - 1) / parts;
        const dim3 grid((unsigned)blocks, (unsigned)parts);
        const uint32_t magic = (uint32_t)((((uint64_t)1 << 32) + units - 1) / units);
        auto dequant = [&](auto whole, auto split) {
            return launch_pdl(parts > 1 ? split : whole, grid, dim3(256), 0, st, 1, tw, tx, blocks0, rpb, piece, units, magic, bits);
        };
        cudaError_t e;
        switch (container_bits(bits)) {
            case 1: e = dequant(dequant_codes_kernel<1, false>, dequant_codes_kernel<1, true>); break;
            case 2: e = dequant(dequant_codes_kernel<2, false>, dequant_codes_kernel<2, true>); break;
            case 4: e = dequant(dequant_codes_kernel<4, false>, dequant_codes_kernel<4, true>); break;
            default: e = dequant(dequant_codes_kernel<8, false>, dequant_codes_kernel<8, true>); break;
        }
        if (e != cudaSuccess) return cuda_fail(e);
    }
    // blocks of up to 128 in rows of whole 128-column groups: the inverse transform runs in the contraction's epilogue,
    // the masked product never reaches memory
    const bool fuse = had_block <= 128 && K % 128 == 0;
    // one gradient: masked product of a and b (see launch_gemm_bf16_masked), then the inverse transform
    const int64_t rows_free = (int64_t)(((uint8_t *)workspace + ws.bytes - (uint8_t *)ws.d1) / (K * 4));
    auto gradient = [&](const void *a, const void *b, int64_t I, int64_t Kc, const uint8_t *mask, void *out, float *d, int opl) {
        Stage gemm_stage(QUEST_STAGE_GEMM, st);
        const int parts = transform_adds_parts(K, had_block) ? divide_contraction(I, K, Kc, rows_free, fuse) : 1;
        if (parts > 1) {                                     // the products run one after the other: both may use d1 and d2
            const int e = launch_gemm_bf16_parts(a, b, I, K, Kc, ws.d1, parts, opl, st);
            return e ? e : launch_iht(ws.d1, I, K, had_block, out, out_dtype, parts, mask, st);
        }
        if (fuse) return launch_gemm_bf16_masked(a, b, I, K, Kc, mask, out, out_dtype, had_block, opl, st);
        const int e = launch_gemm_bf16_masked(a, b, I, K, Kc, mask, d, QUEST_F32, 0, opl, st);
        return e ? e : launch_iht(d, I, K, had_block, out, out_dtype, 1, nullptr, st);
    };
    // activation gradient of Algorithm 2 with its trust mask: d1[m][k] = M_x[m][k] * sum_n dy[m][n] wq_h[n][k]
    if (dx && (s = gradient(dy, ws.wh, M, N, mx, dx, ws.d1, 1))) return s;
    // weight gradient of Algorithm 2 with its trust mask: d2[n][k] = M_w[n][k] * sum_m dy[m][n] xq_h[m][k]
    if (dw && (s = gradient(dy, ws.xh, N, M, mw, dw, ws.d2, 2))) return s;
    return QUEST_OK;
}
