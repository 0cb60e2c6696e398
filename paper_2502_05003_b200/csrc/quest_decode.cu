// The inference layer with cached weights for a handful of rows of x (decoding): y = (xq cw^T) sx sw for M <= 32.
//
// The tensor-core kernel of quest_gemm.cu gives such a layer 256 x 128 tiles of CTA pairs, of which 8 to 32 rows are wanted:
// 16 pairs for 2048 columns (8.2 us with the quantizer; 11.7 with the single-CTA 128 x 256 tiles it had when this was
// written).  What bounds the work is reading w once
// (4 MB at 2048 x 2048: under a microsecond from HBM) and latency, so here a CTA takes 16, 32 or 48 rows of w, its eight
// warps split K, and every warp multiplies with mma.sync m16n8k32 (w is the 16-row operand, the rows of x are the 8
// columns): integer sums are exact in any order, so the K positions a lane holds are simply 16 consecutive bytes of
// its row.  A lane copies its own bytes with cp.async into its own slots of a ring (no barrier in the main loop, up
// to eight chunks in flight: loads into registers left the warps waiting for every chunk in turn, 14.6 us for 30 MB
// of w against 9.0).  The partial sums of the eight warps meet in shared memory.  tcgen05 would need 128-row tiles,
// tensor memory and descriptors for a product whose arithmetic is not what takes the time.
// Whole layer at 2048 x 2048, device time back to back over eight layers: one row 11.7 -> 3.7 us, 32 rows 12.0 -> 5.2 us;
// 24 rows x 5504 x 2048 from packed codes 16.6 -> 8.8 us.
//
// Two forms.  FUSED (few rows): the CTA rotates and quantizes x itself while its first loads of w are in flight;
// every CTA repeats that work, one launch does the layer.  Otherwise the quantizer is a launch of its own, and this
// kernel requests its part of w before it waits for it.
//
// w comes either as the operand that an earlier call left in the workspace, or as packed codes, which are unpacked
// on the way to the tensor cores and also written to the workspace as the operand that later calls may reuse.
//
// Compiled with -fmad=false; the rotation, the row's RMS, the projection and the trust test follow the operation order
// stated in quest_quantize.cu bit for bit (rows with NaN or infinities included).
#include <cuda_bf16.h>

#include <type_traits>

#include "quest_internal.cuh"
#include "quest_operand.cuh"

namespace quest {
namespace {

constexpr int WARPS = 8;
constexpr int THREADS = 32 * WARPS;
constexpr int MAX_TASKS = 2;              // FUSED: 256-element pieces of x per warp
constexpr int FUSED_ROWS = 8;

struct DecodeArgs {
    const void *x;
    int x_f32, M, N, K, bits, g;
    QuantConsts qc;
    uint8_t *codes;                       // FUSED: outputs of the quantizer
    float *scales;
    uint8_t *mask;
    const uint8_t *wq;                    // packed codes of w (SRC_CODES*)
    int8_t *b8;                           // operand of w in the workspace: read (SRC_OP*), written (SRC_CODES*)
    int32_t *rs_b;                        // its row sums (8-bit codes)
    const float *sw;
    const int8_t *a8;                     // not FUSED: operand, row sums and scales of x
    const int32_t *rs_a;
    const float *sx;
    void *y;
    int y_f32;
    float fold;                           // exact power of two of the operand scaling, applied to the row scale ...
    int shift;                            // ... or to the sums: where the contraction of many rows does which
    int pitch;                            // FUSED: bytes per row of the operand of x in shared memory
};

enum { SRC_OP8 = 0, SRC_OP4 = 1, SRC_CODES1 = 2, SRC_CODES2 = 3, SRC_CODES4 = 4, SRC_CODES8 = 5 };
// words that 16 elements take in the source
template <int SRC> struct SrcWords { static constexpr int N = SRC == SRC_OP8 || SRC == SRC_CODES8 ? 4 : SRC == SRC_OP4 || SRC == SRC_CODES4 ? 2 : 1; };

// Eight E2M1 nibbles of the one- and two-bit grids (0x2, 0xA: +-1; 0x5, 0xD: +-3) -> eight bytes 16 c, the even
// elements in one word and the odd ones in the other (x is put in the same order).  16 c has the nibble
// (s, s, s ^ m0, 1) on top: s the sign bit, m0 the lowest bit of the E2M1 code.
__device__ __forceinline__ void bytes_of_e2m1(uint32_t w, uint32_t &even, uint32_t &odd) {
    const uint32_t o = (w & 0x88888888u) | ((w >> 1) & 0x44444444u) | (((w << 1) ^ (w >> 2)) & 0x22222222u) | 0x11111111u;
    even = (o << 4) & 0xF0F0F0F0u;
    odd = o & 0xF0F0F0F0u;
}

// BYTES (4, 8 or 16) from global to this thread's slot, zeros where `ok` is false (nothing is read then).
template <int BYTES>
__device__ __forceinline__ void copy_async(uint32_t slot, const void *src, bool ok) {
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(slot), "l"(src), "r"(ok ? 16 : 0) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;" ::"r"(slot), "l"(src), "r"(ok ? BYTES : 0), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// 16 elements of a row of w from position k, as the source stores them, to a slot.
template <int SRC>
__device__ __forceinline__ void fetch_w(const DecodeArgs &a, int row, int k, uint8_t *slot) {
    const bool ok = row < a.N && k < a.K;
    const long long e = ok ? (long long)row * a.K + k : 0;
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(slot);
    if constexpr (SRC == SRC_OP8) copy_async<16>(s, a.b8 + e, ok);
    else if constexpr (SRC == SRC_CODES8) copy_async<16>(s, a.wq + e, ok);
    else if constexpr (SRC == SRC_OP4) copy_async<8>(s, a.b8 + (e >> 1), ok);
    else if constexpr (SRC == SRC_CODES4) copy_async<8>(s, a.wq + (e >> 1), ok);
    else if constexpr (SRC == SRC_CODES2) copy_async<4>(s, a.wq + (e >> 2), ok);
    else *reinterpret_cast<uint32_t *>(slot) = ok ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(a.wq + (e >> 3))) : 0u;
}

// Words of a slot -> 16 operand bytes; packed codes also leave as the operand later calls read from the workspace.
// Elements past the row (k >= K) meet zeros of x, so what they become does not matter.
template <int SRC>
__device__ __forceinline__ void operand_w(const DecodeArgs &a, int row, int k, const uint32_t (&r)[SrcWords<SRC>::N],
                                          uint32_t (&o)[4], int &rsum) {
    constexpr int NW = SrcWords<SRC>::N;
    const bool ok = row < a.N && k < a.K;
    const long long e = (long long)row * a.K + k;
    if constexpr (SRC == SRC_OP8) {
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = r[i];
    } else if constexpr (SRC == SRC_OP4) {
        bytes_of_e2m1(r[0], o[0], o[1]);
        bytes_of_e2m1(r[NW - 1], o[2], o[3]);
    } else if constexpr (SRC == SRC_CODES8 || SRC == SRC_CODES4) {
        operand16_from_codes<SRC == SRC_CODES8 ? 8 : 4>(r, a.bits, o);
        if (SRC == SRC_CODES8 && a.rs_b) {
#pragma unroll
            for (int i = 0; i < 4; ++i) rsum = ok ? __dp4a((int)o[i], 0x01010101, rsum) : rsum;
        }
        if (ok) *reinterpret_cast<uint4 *>(a.b8 + e) = make_uint4(o[0], o[1], o[2], o[3]);
    } else {
        constexpr int CB = SRC == SRC_CODES1 ? 1 : 2;
        const uint32_t n0 = e2m1_word_from_levels<CB>(r[0] & (CB == 1 ? 0xFFu : 0xFFFFu));
        const uint32_t n1 = e2m1_word_from_levels<CB>((r[0] >> (8 * CB)) & (CB == 1 ? 0xFFu : 0xFFFFu));
        bytes_of_e2m1(n0, o[0], o[1]);
        bytes_of_e2m1(n1, o[2], o[3]);
        if (ok) *reinterpret_cast<uint2 *>(a.b8 + (e >> 1)) = make_uint2(n0, n1);
    }
}

__device__ __forceinline__ void mma_s8(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// FUSED: rotates and quantizes the M rows of x.  A task is 256 consecutive elements of a row, eight to a lane; the
// warps share the tasks, the rotated elements stay in registers across the barrier that the row's RMS needs.
__device__ __forceinline__ void quantize_rows_in_cta(const DecodeArgs &a, int8_t *xop, float *xs, float *part, float *s_sx,
                                                     int *s_rsa) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nch = (a.K + 255) >> 8;
    const int tasks = a.M * nch;
    const int g = a.g;
    float v[MAX_TASKS][8];
#pragma unroll
    for (int i = 0; i < MAX_TASKS; ++i) {
        const int q = warp + WARPS * i;
        const int row = q / nch, e0 = (q - row * nch) * 256 + lane * 8;
        if (q < tasks && e0 < a.K) {
            if (a.x_f32) {
                const float4 *src = reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(a.x) + (long long)row * a.K + e0);
                const float4 lo = __ldg(src), hi = __ldg(src + 1);
                v[i][0] = lo.x; v[i][1] = lo.y; v[i][2] = lo.z; v[i][3] = lo.w;
                v[i][4] = hi.x; v[i][5] = hi.y; v[i][6] = hi.z; v[i][7] = hi.w;
            } else {
                const uint4 w = __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const uint16_t *>(a.x) + (long long)row * a.K + e0));
                const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    v[i][2 * j] = __uint_as_float(ww[j] << 16);
                    v[i][2 * j + 1] = __uint_as_float(ww[j] & 0xFFFF0000u);
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[i][j] = 0.0f;
        }
    }
    // rotation, descending stride: partners in other tasks through shared memory (blocks of 512 and more) ...
    for (int h = g >> 1; h >= 256; h >>= 1) {
        const int d = h >> 8;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < MAX_TASKS; ++i) {
            const int q = warp + WARPS * i;
            if (q < tasks) {
                float4 *dst = reinterpret_cast<float4 *>(xs + q * 256 + lane * 8);
                dst[0] = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
                dst[1] = make_float4(v[i][4], v[i][5], v[i][6], v[i][7]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < MAX_TASKS; ++i) {
            const int q = warp + WARPS * i;
            if (q < tasks) {
                const int row = q / nch, c = q - row * nch;
                const float4 *src = reinterpret_cast<const float4 *>(xs + (row * nch + (c ^ d)) * 256 + lane * 8);
                const float4 lo = src[0], hi = src[1];
                const float o[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                const float sg = (c & d) ? -1.0f : 1.0f;
#pragma unroll
                for (int j = 0; j < 8; ++j) v[i][j] = __fmaf_rn(v[i][j], sg, o[j]);
            }
        }
    }
    // ... in other lanes by shuffles, then inside the lane
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1)
        if (8 * d < g) {
            const float sg = (lane & d) ? -1.0f : 1.0f;
#pragma unroll
            for (int i = 0; i < MAX_TASKS; ++i)
                if (warp + WARPS * i < tasks) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[i][j] = __fmaf_rn(v[i][j], sg, __shfl_xor_sync(0xffffffffu, v[i][j], d));
                }
        }
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1)
        if (h < g) {
#pragma unroll
            for (int i = 0; i < MAX_TASKS; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if ((j & h) == 0) {
                        const float p = v[i][j], q = v[i][j + h];
                        v[i][j] = __fadd_rn(p, q);
                        v[i][j + h] = __fsub_rn(p, q);
                    }
        }
    // sum of squares: pairwise in the lane, over the lanes of the task, over the tasks of the (zero-padded) row
#pragma unroll
    for (int i = 0; i < MAX_TASKS; ++i) {
        const int q = warp + WARPS * i;
        float s[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) s[j] = __fmul_rn(v[i][j], v[i][j]);
        float ss = __fadd_rn(__fadd_rn(__fadd_rn(s[0], s[1]), __fadd_rn(s[2], s[3])),
                             __fadd_rn(__fadd_rn(s[4], s[5]), __fadd_rn(s[6], s[7])));
#pragma unroll
        for (int m = 1; m < 32; m <<= 1) ss = __fadd_rn(ss, __shfl_xor_sync(0xffffffffu, ss, m));
        if (lane == 0 && q < tasks) part[q] = ss;
    }
    __syncthreads();
    const bool writer = blockIdx.x == 0;                       // every CTA computes the same bits, one stores them
    const int cb = container_bits(a.bits);
    // operand bytes 2^(7-b) c, or k - 128 at 8 bits, as in operand16_from_codes
    const uint32_t op_m = ((0xFFu << (8 - a.bits)) & 0xFFu) * 0x01010101u;
    const uint32_t op_c = a.bits == 8 ? 0x80808080u : (0x80u | (1u << (7 - a.bits))) * 0x01010101u;
#pragma unroll
    for (int i = 0; i < MAX_TASKS; ++i) {
        const int q = warp + WARPS * i;
        if (q < tasks) {
            const int row = q / nch, c = q - row * nch, e0 = c * 256 + lane * 8;
            float ss = lane < nch ? part[row * nch + lane] : 0.0f;
#pragma unroll
            for (int m = 1; m < 32; m <<= 1) ss = __fadd_rn(ss, __shfl_xor_sync(0xffffffffu, ss, m));
            const float rms = __fsqrt_rn(__fdiv_rn(ss, (float)a.K));
            const float inv = (rms > 0.0f) ? __fdiv_rn(a.qc.A, rms) : 0.0f;
            if (c == 0 && lane == 0) {
                const float sx = __fmul_rn(rms, a.qc.B);
                s_sx[row] = sx;
                if (writer) a.scales[row] = sx;
            }
            // levels as bytes: the rounding constant leaves each level in the low bits of its sum
            uint32_t kb[2] = {0u, 0u};
#pragma unroll
            for (int j = 7; j >= 0; --j) {
                const float t = __fmaf_rn(v[i][j], inv, a.qc.c0);
                const float km = __fadd_rn(fminf(fmaxf(t, 0.0f), a.qc.top), 12582912.0f);
                kb[j >> 2] = (kb[j >> 2] << 8) + (__float_as_uint(km) - 0x4B400000u);
            }
            const uint32_t op[2] = {lop3_mask_xor_set(kb[0] << (8 - a.bits), op_m, op_c),
                                    lop3_mask_xor_set(kb[1] << (8 - a.bits), op_m, op_c)};
            int rs = __dp4a((int)op[0], 0x01010101, __dp4a((int)op[1], 0x01010101, 0));
            if (e0 < a.K) {
                *reinterpret_cast<uint2 *>(xop + row * a.pitch + e0) = make_uint2(op[0], op[1]);
                if (writer) {
                    uint32_t mbits = 0;
                    uint64_t packed = 0;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const uint32_t k = (kb[j >> 2] >> (8 * (j & 3))) & 0xFFu;
                        const float t = __fmaf_rn(v[i][j], inv, a.qc.c0);
                        // not "<=": a position that is not a number counts as trusted, as in the sign tests of quest_quantize.cu
                        mbits |= (fabsf(__fsub_rn(t, (float)k)) > a.qc.h ? 0u : 1u) << j;
                        packed |= (uint64_t)k << (j * cb);
                    }
                    uint8_t *dst = a.codes + ((long long)row * a.K + e0) / 8 * cb;
                    if (cb == 8) *reinterpret_cast<uint2 *>(dst) = make_uint2((uint32_t)packed, (uint32_t)(packed >> 32));
                    else if (cb == 4) *reinterpret_cast<uint32_t *>(dst) = (uint32_t)packed;
                    else if (cb == 2) *reinterpret_cast<uint16_t *>(dst) = (uint16_t)packed;
                    else *dst = (uint8_t)packed;
                    if (a.mask) a.mask[((long long)row * a.K + e0) >> 3] = (uint8_t)mbits;
                }
            } else {
                rs = 0;
            }
            if (a.bits == 8) {
#pragma unroll
                for (int m = 1; m < 32; m <<= 1) rs += __shfl_xor_sync(0xffffffffu, rs, m);
                if (lane == 0) atomicAdd(&s_rsa[row], rs);     // integers: any order
            }
        }
    }
}

// DEEP: the CTA has an SM to itself.
template <bool FUSED, int MT, int NT, bool DEEP> struct Ring {
    static constexpr int UNITS = 2 * MT + (FUSED ? 0 : NT);            // 16-byte slots per thread and chunk
    static constexpr int STAGE = UNITS * THREADS * 16;
    static constexpr int MOST = DEEP ? 48 : 24;                        // chunks in flight: at most 96 KB where two CTAs share an SM
    static constexpr int DEPTH = MOST / UNITS > 8 ? 8 : MOST / UNITS;
    static constexpr int RED = WARPS * 8 * NT * 16 * MT * 4;           // the partial sums take the ring's place
    static constexpr int BYTES = DEPTH * STAGE > RED ? DEPTH * STAGE : RED;
};

template <int SRC, bool FUSED, int MT, int NT, bool DEEP>
__global__ void __launch_bounds__(THREADS, DEEP ? 1 : 2)
decode_kernel(const __grid_constant__ DecodeArgs a) {
    using L = Ring<FUSED, MT, NT, DEEP>;
    constexpr int ROWS = 16 * MT;
    constexpr int NW = SrcWords<SRC>::N;
    constexpr int D = L::DEPTH;
    constexpr bool SPLIT = SRC == SRC_OP4 || SRC == SRC_CODES1 || SRC == SRC_CODES2;  // even and odd elements apart (bytes_of_e2m1)
    extern __shared__ __align__(16) uint8_t smem[];
    int *red = reinterpret_cast<int *>(smem);                          // [WARPS][8 NT][ROWS], after the main loop
    __shared__ float part[WARPS * MAX_TASKS];
    __shared__ float s_sx[FUSED_ROWS];
    __shared__ int s_rsa[FUSED_ROWS];
    __shared__ int s_rsb[SRC == SRC_CODES8 ? WARPS * ROWS : 1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gq = lane >> 2, t = lane & 3;
    const int r0 = (int)blockIdx.x * ROWS;
    // chunks of 64 elements of K, dealt to the warps two neighbours at a time (whole 128-byte lines of a byte operand)
    const int nc = (a.K + 63) >> 6;
    auto chunk = [&](int j) { return 2 * WARPS * (j >> 1) + 2 * warp + (j & 1); };
    auto slot = [&](int j, int u) { return smem + ((j % D) * L::UNITS + u) * (THREADS * 16) + tid * 16; };
    auto fetch_w_chunk = [&](int j) {
        const int k = chunk(j) * 64 + 16 * t;
#pragma unroll
        for (int u = 0; u < 2 * MT; ++u) fetch_w<SRC>(a, r0 + 8 * u + gq, k, slot(j, u));
    };
    auto fetch_x_chunk = [&](int j) {
        if constexpr (!FUSED) {
            const int k = chunk(j) * 64 + 16 * t;
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                const int xr = 8 * n + gq;
                const bool ok = xr < a.M && k < a.K;
                const long long e = ok ? (long long)xr * a.K + k : 0;
                const uint32_t s = (uint32_t)__cvta_generic_to_shared(slot(j, 2 * MT + n));
                copy_async<16>(s, a.a8 + e, ok);
            }
        }
    };
    // FUSED: everything this kernel reads may come from the previous one.  Otherwise the previous kernel is the quantizer
    // of this call, which lets this one start only after its own predecessors have finished: w may be read at once.
    if constexpr (FUSED) pdl_wait();
    pdl_launch_dependents();
#pragma unroll 1
    for (int j = 0; j < D; ++j) {
        if (chunk(j) < nc) fetch_w_chunk(j);
        if constexpr (FUSED) copy_commit();
    }
    int8_t *xop = reinterpret_cast<int8_t *>(smem + L::BYTES);
    if constexpr (FUSED) {
        if (tid < FUSED_ROWS) s_rsa[tid] = 0;
        float *xs = reinterpret_cast<float *>(xop + (size_t)a.M * a.pitch);
        if (a.bits == 8) __syncthreads();
        quantize_rows_in_cta(a, xop, xs, part, s_sx, s_rsa);
        __syncthreads();
    } else {
        pdl_wait();
#pragma unroll 1
        for (int j = 0; j < D; ++j) {                                  // one group per chunk, w's share in the first
            if (chunk(j) < nc) fetch_x_chunk(j);
            copy_commit();
        }
    }
    int acc[MT][NT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[m][n][i] = 0;
    int rsum[MT][2] = {};
#pragma unroll 1
    for (int j = 0; chunk(j) < nc; ++j) {                              // uniform over the warp
        copy_wait<D - 1>();                                            // this thread's own copies of chunk j have landed
        const int k = chunk(j) * 64 + 16 * t;
        uint32_t o[MT][2][4];
#pragma unroll
        for (int u = 0; u < 2 * MT; ++u) {
            uint32_t raw[NW];
            const uint8_t *sl = slot(j, u);
            if constexpr (NW == 4) {
                const uint4 v = *reinterpret_cast<const uint4 *>(sl);
                raw[0] = v.x; raw[1] = v.y; raw[2] = v.z; raw[NW - 1] = v.w;
            } else if constexpr (NW == 2) {
                const uint2 v = *reinterpret_cast<const uint2 *>(sl);
                raw[0] = v.x; raw[NW - 1] = v.y;
            } else {
                raw[0] = *reinterpret_cast<const uint32_t *>(sl);
            }
            operand_w<SRC>(a, r0 + 8 * u + gq, k, raw, o[u >> 1][u & 1], rsum[u >> 1][u & 1]);
        }
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            uint32_t b[4] = {0u, 0u, 0u, 0u};
            if constexpr (FUSED) {
                const int xr = 8 * n + gq;
                if (xr < a.M && k < a.K) {
                    const uint4 w = *reinterpret_cast<const uint4 *>(xop + xr * a.pitch + k);
                    b[0] = w.x; b[1] = w.y; b[2] = w.z; b[3] = w.w;
                }
            } else {
                const uint4 w = *reinterpret_cast<const uint4 *>(slot(j, 2 * MT + n));
                b[0] = w.x; b[1] = w.y; b[2] = w.z; b[3] = w.w;
            }
            if constexpr (SPLIT) {
#pragma unroll
                for (int q = 0; q < 4; q += 2) {
                    const uint32_t e = __byte_perm(b[q], b[q + 1], 0x6420), d = __byte_perm(b[q], b[q + 1], 0x7531);
                    b[q] = e;
                    b[q + 1] = d;
                }
            }
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                mma_s8(acc[m][n], o[m][0][0], o[m][1][0], o[m][0][1], o[m][1][1], b[0], b[1]);
                mma_s8(acc[m][n], o[m][0][2], o[m][1][2], o[m][0][3], o[m][1][3], b[2], b[3]);
            }
        }
        if (chunk(j + D) < nc) {                                       // the slots just read
            fetch_w_chunk(j + D);
            fetch_x_chunk(j + D);
        }
        copy_commit();
    }
    copy_wait<0>();
    __syncthreads();                                                   // every warp has left the ring
    // partial sums of the eight K slices
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                red[(warp * 8 * NT + 8 * n + 2 * t + (i & 1)) * ROWS + 16 * m + 8 * (i >> 1) + gq] = acc[m][n][i];
    if constexpr (SRC == SRC_CODES8) {
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                int s = rsum[m][h];
                s += __shfl_xor_sync(0xffffffffu, s, 1);
                s += __shfl_xor_sync(0xffffffffu, s, 2);
                if (t == 0) s_rsb[warp * ROWS + 16 * m + 8 * h + gq] = s;
            }
    }
    __syncthreads();
    if (SRC == SRC_CODES8 && a.rs_b && tid < ROWS && r0 + tid < a.N) {
        int s = 0;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) s += s_rsb[w * ROWS + tid];
        a.rs_b[r0 + tid] = s;
    }
    for (int o = tid; o < ROWS * a.M; o += THREADS) {
        const int n = o / ROWS, r = o - n * ROWS, col = r0 + r;
        if (col >= a.N) continue;
        int s = 0;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) s += red[(w * 8 * NT + n) * ROWS + r];
        if (a.bits == 8) {                                             // c = 2v + 1 on both sides
            int rb;
            if constexpr (SRC == SRC_CODES8) {
                rb = 0;
#pragma unroll
                for (int w = 0; w < WARPS; ++w) rb += s_rsb[w * ROWS + r];
            } else {
                rb = __ldg(a.rs_b + col);
            }
            s = (int)(4u * (uint32_t)s + 2u * (uint32_t)(FUSED ? s_rsa[n] : __ldg(a.rs_a + n)) + 2u * (uint32_t)rb + (uint32_t)a.K);
        }
        s >>= a.shift;
        const float sxr = __fmul_rn(FUSED ? s_sx[n] : __ldg(a.sx + n), a.fold);
        const float yv = __fmul_rn(__fmul_rn(sxr, __ldg(a.sw + col)), (float)s);
        if (a.y_f32) reinterpret_cast<float *>(a.y)[(long long)n * a.N + col] = yv;
        else reinterpret_cast<__nv_bfloat16 *>(a.y)[(long long)n * a.N + col] = __float2bfloat16_rn(yv);
    }
}

template <int SRC, bool FUSED, int MT, int NT, bool DEEP = false>
cudaError_t launch_one(const DecodeArgs &a, cudaStream_t st) {
    size_t smem = Ring<FUSED, MT, NT, DEEP>::BYTES;
    const int ctas = (a.N + 16 * MT - 1) / (16 * MT);
    if (FUSED) smem += (size_t)a.M * a.pitch + (a.g >= 512 ? (size_t)a.M * ((a.K + 255) / 256) * 1024 : 0);
    if ((DEEP || (SRC == SRC_CODES8 && !FUSED && ctas <= num_sms())) && smem < 116 * 1024) smem = 116 * 1024;      // one CTA per SM
    static DynamicSmemOnce once;
    const cudaError_t e = once.set(decode_kernel<SRC, FUSED, MT, NT, DEEP>, DEEP ? 200 * 1024 : 144 * 1024);
    if (e != cudaSuccess) return e;
    return launch_pdl(decode_kernel<SRC, FUSED, MT, NT, DEEP>, dim3((unsigned)ctas), dim3(THREADS), smem, st, 1, a);
}

template <int SRC, bool FUSED>
cudaError_t launch_src(const DecodeArgs &a, bool two, cudaStream_t st) {
    if constexpr (FUSED) {
        return two ? launch_one<SRC, true, 2, 1>(a, st) : launch_one<SRC, true, 1, 1>(a, st);
    } else {
        // One CTA per SM, with up to twice the chunks in flight, where 16, 32 or 48 rows of w a CTA allow it: started while the
        // quantizer drains, two would share each SM that is free first, and a second CTA on some SMs is what all wait for.
        // 24 x 5504 x 2048 from packed codes 10.9 -> 8.9 us, with w's operand prepared 9.2 -> 8.3; 24 x 2048 x 5504 10.0 -> 9.4 and
        // 8.7 -> 8.3 .. 8.7; 5 x 5504 x 2048 from codes 8.0 -> 6.7; 32 x 5504 x 5504 15.0 -> 13.2 (back to back over 40 layers); equal
        // up to 160 elements a row.  Packed codes of 8 bits gain the single CTA
        // only (5 x 5504 x 2048 with 48 rows 7.6 -> 8.2); one and two bits are held by unpacking and lose a little even there
        // (24 x 4096 x 4096 at two bits 8.5 -> 8.7).
        if constexpr (SRC == SRC_OP8 || SRC == SRC_CODES4) {
            const int mt = (a.N + 16 * num_sms() - 1) / (16 * num_sms());
            auto deep = [&](auto nt) {
                constexpr int NT = decltype(nt)::value;
                return mt == 1 ? launch_one<SRC, false, 1, NT, true>(a, st) : mt == 2 ? launch_one<SRC, false, 2, NT, true>(a, st)
                                                                                    : launch_one<SRC, false, 3, NT, true>(a, st);
            };
            if (mt <= 3)
                return a.M <= 8 ? deep(std::integral_constant<int, 1>()) : a.M <= 16 ? deep(std::integral_constant<int, 2>())
                                                                                     : deep(std::integral_constant<int, 4>());
            return a.M <= 8 ? launch_one<SRC, false, 2, 1>(a, st) : a.M <= 16 ? launch_one<SRC, false, 2, 2>(a, st)
                                                                              : launch_one<SRC, false, 2, 4>(a, st);
        } else {
            if (a.M <= 8) return two ? launch_one<SRC, false, 2, 1>(a, st) : launch_one<SRC, false, 1, 1>(a, st);
            if (a.M <= 16) return two ? launch_one<SRC, false, 2, 2>(a, st) : launch_one<SRC, false, 1, 2>(a, st);
            return two ? launch_one<SRC, false, 2, 4>(a, st) : launch_one<SRC, false, 1, 4>(a, st);
        }
    }
}

template <bool FUSED>
cudaError_t launch_form(int src, const DecodeArgs &a, bool two, cudaStream_t st) {
    switch (src) {
        case SRC_OP8: return launch_src<SRC_OP8, FUSED>(a, two, st);
        case SRC_OP4: return launch_src<SRC_OP4, FUSED>(a, two, st);
        case SRC_CODES1: return launch_src<SRC_CODES1, FUSED>(a, two, st);
        case SRC_CODES2: return launch_src<SRC_CODES2, FUSED>(a, two, st);
        case SRC_CODES4: return launch_src<SRC_CODES4, FUSED>(a, two, st);
        default: return launch_src<SRC_CODES8, FUSED>(a, two, st);
    }
}

}  // namespace

// Where the decoding path serves.  Its time grows in steps with N, with the CTAs that share an SM (a CTA takes 16 rows of
// w, 32 above 16 per SM; from 32 rows per SM on CTAs begin to share one, above 64 there is a second round; from the byte
// operand and 4-bit codes a CTA of 16, 32 or 48 rows has an SM to itself up to 48 rows per SM, and these limits, measured
// when it had not, were not moved), with the
// groups of eight rows of x, and at one and two bits with the unpacking of w to bytes, which the FP4 contraction of
// quest_gemm.cu need not do.  Against that contraction (device time back to back, us, here / there):
//    4 bits, operand: 8 x 32768 x 4096 27.1 / 41.0; 32 x 4096 x 4096 10.0 / 10.5, 32 x 11008 x 512 1.09 of it, 32 x 16384 x
//                     2048 14.3 / 12.5;  codes: 32 x 32768 x 2048 32.2 / 42.7  (8 bits behave as 4)
//    1 bit, operand:  8 x 8192 x 8192 0.9 of it, 8 x 16384 x 2048 10.7 / 10.7, x 4096 15.9 / 12.9; 16 x 5504 x 8192 1.16;
//                     32 x 2368 x 4096 1.28, 32 x 5504 x 1024 1.09
//    2 bits, codes:   8 x 9472 x 4096 13.8 / 16.4, 8 x 11008 x 4096 18.7 / 18.2, 8 x 32768 x 4096 39.5 / 42.5
// (the contraction of a large w varies by a quarter with what L2 holds: a limit is where it is ahead all the same).
bool decode_serves(int64_t M, int64_t N, int64_t K, int bits, bool w_codes) {
    if (M < 1 || N < 1 || M > 32) return false;
    const int64_t sms = num_sms();
    if (bits > 2) return w_codes || M <= 16 || N <= 64 * sms || (N <= 96 * sms && K >= 1024);
    if (bits == 2 && w_codes && M <= 8 && N > 96 * sms) return true;
    // longest rows at one and two bits; columns: up to 8, below 16, 32, 48, up to 64, 96 rows of w per SM, and more
    constexpr int ALL = 16384;
    static constexpr int LIMIT[2][3][7] = {
        // operand in the workspace: up to 8, 16, 32 rows of x
        {{ALL, ALL, ALL, ALL, ALL, 3072, 1024}, {ALL, ALL, 8192, 5504, 8192, 1536, 0}, {ALL, 2048, 1024, 0, 0, 0, 0}},
        // packed codes
        {{ALL, ALL, ALL, ALL, ALL, 4096, 3072}, {ALL, ALL, 8192, 5504, 8192, 2048, 1024}, {ALL, 3072, 2048, 1024, 1024, 0, 0}}};
    const int col = N <= 8 * sms ? 0 : N < 16 * sms ? 1 : N < 32 * sms ? 2 : N < 48 * sms ? 3 : N <= 64 * sms ? 4 : N <= 96 * sms ? 5 : 6;
    return K <= LIMIT[w_codes ? 1 : 0][M <= 8 ? 0 : M <= 16 ? 1 : 2][col];
}

// Quantizing in every CTA saves a launch: 2.7 us of host time, and the dependency between the two.  It pays on the
// device while a warp has one piece of x and the CTAs are resident at once (two launches take 1.0 .. 1.2 times as long
// back to back up to 32 rows of w per SM, 0.85 .. 1.1 up to 64; with a second round of CTAs, which quantize again, 0.65
// .. 0.9).  With two pieces per warp two launches are the faster device work (0.85 .. 0.9 of one at 1 x 2048 x 4096 and
// 2 x 2048 x 2048, 0.83 at 4 x 2048 x 1024), which only a replayed graph would see; a program that issues its calls
// waits for the host (the same three 0.95 .. 1.05, 1.02 and 1.1), so they are fused up to 32 rows per SM.
bool decode_fuses_quantizer(int64_t M, int64_t N, int64_t K) {
    const int64_t pieces = M * ((K + 255) / 256), sms = num_sms();
    return M <= FUSED_ROWS && (pieces <= WARPS ? N <= 64 * sms : pieces <= WARPS * MAX_TASKS && N < 32 * sms);
}

int launch_decode(const QuantJob &jx, int dtype, bool fused, const uint8_t *wq, int8_t *b8, int32_t *rs_b, const float *sw,
                  bool w_codes, int64_t N, int64_t K, int bits, int had_block, float trust_factor, void *y, int y_dtype,
                  cudaStream_t st) {
    DecodeArgs a;
    a.x = jx.x; a.x_f32 = dtype == QUEST_F32; a.M = (int)jx.rows; a.N = (int)N; a.K = (int)K; a.bits = bits; a.g = had_block;
    a.qc = make_quant_consts(bits, had_block, trust_factor);
    a.codes = jx.codes; a.scales = jx.scales; a.mask = jx.mask;
    a.wq = wq; a.b8 = b8; a.rs_b = bits == 8 ? rs_b : nullptr; a.sw = sw;
    a.a8 = jx.op8; a.rs_a = jx.rowsum; a.sx = jx.scales;
    a.y = y; a.y_f32 = y_dtype == QUEST_F32;
    const bool e4 = e2m1_operands(bits, bits);
    // operand scalings: 2^(7-b) c on both sides, 16 c for w of one or two bits (bytes_of_e2m1).  The contraction of
    // quest_gemm.cu takes its power of two out of the row scale, and has none at one and two bits (E2M1 operands):
    // there the sums are shifted, or products of scales below 2^-116 would lose bits that it keeps.
    a.fold = bits == 8 || e4 ? 1.0f : 1.0f / (float)(1 << (14 - 2 * bits));
    a.shift = e4 ? 11 - bits : 0;
    a.pitch = (int)((K + 127) / 128 * 128 + 64);               // rows 64 bytes apart modulo 128: two rows of a load share no bank
    int src = e4 ? SRC_OP4 : SRC_OP8;
    if (w_codes) {
        const int cb = container_bits(bits);
        src = cb == 1 ? SRC_CODES1 : cb == 2 ? SRC_CODES2 : cb == 4 ? SRC_CODES4 : SRC_CODES8;
    }
    // 32 rows of w per CTA once 16 would give more CTAs than there are SMs: half the reads (or quantizations) of x.  (The
    // byte operand and 4-bit codes behind a quantizer launch follow launch_src instead, up to 48 rows per SM.)
    const bool two = N > 16ll * num_sms();
    const cudaError_t e = fused ? launch_form<true>(src, a, two, st) : launch_form<false>(src, a, two, st);
    return e == cudaSuccess ? QUEST_OK : cuda_fail(e);
}

}  // namespace quest
