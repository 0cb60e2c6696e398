// Internal declarations shared by the translation units of the library (not part of the ABI).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "quest.h"

namespace quest {

// alpha*(b), b = 1..8 (Section 3.1): minimiser of the Gaussian quantisation MSE on the
// 2^b-point grid, rounded to binary32.
__host__ __device__ inline float alpha_star(int bits) {
    switch (bits) {
        case 1: return 0.7978846f;
        case 2: return 1.4935300f;
        case 3: return 2.0510680f;
        case 4: return 2.5140045f;
        case 5: return 2.9161513f;
        case 6: return 3.2779846f;
        case 7: return 3.6110970f;
        case 8: return 3.9222038f;
        default: return 0.0f;
    }
}

__host__ __device__ inline int container_bits(int bits) {
    return bits == 1 ? 1 : bits == 2 ? 2 : bits <= 4 ? 4 : 8;
}

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Per-row constants of the projection, computed once on the host in binary32.
struct QuantConsts {
    float c0;      // (2^b-1)/2: centre of the level axis
    float top;     // 2^b-1: highest level
    float A;       // (2^b-1)/(2 alpha*): RMS-normalised value -> level-axis slope
    float B;       // alpha*/((2^b-1) sqrt(g)): RMS of the un-normalised rotation -> scale
    float h;       // trust_factor/2: trust bound in level steps (FP4 grid: trust_factor, in E2M1 value units)
    float hi;      // the largest binary32 number that is at most top + h
};
QuantConsts make_quant_consts(int bits, int had_block, float trust_factor);

// Rounding grids: the uniform zero-free grid of Eq. 1, or the FP4 (E2M1) grid of Section 4.4.
enum { GRID_UNIFORM = 0, GRID_FP4 = 1 };
// alpha*_FP4: minimiser of the Gaussian quantisation MSE on the E2M1 grid scaled to [-1, 1].
__host__ __device__ inline float alpha_star_fp4() { return 2.9224751f; }

// Operand layout of the int8 tensor-core contraction inside the workspace.
struct Workspace {
    int8_t *a8;        // [M x K] int8 operand values of x
    int8_t *b8;        // [N x K] int8 operand values of w
    int32_t *rs_a;     // [M] row sums of a8 (used only with 8-bit codes)
    int32_t *rs_b;     // [N]
    size_t bytes;
};
Workspace carve_workspace(void *base, int64_t M, int64_t N, int64_t K);

// Programmatic dependent launch.  Every kernel of the library is launched with the
// programmatic-stream-serialization attribute and (1) lets the next kernel in the stream begin
// its launch and set-up early, (2) waits for the previous kernel's grid to complete and flush
// before it touches global memory.  The wait is what keeps stream order; launched without the
// attribute both instructions are no-ops.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// HOLD: the next kernel may begin only once everything before this one has finished.  A template parameter: with the
// choice read from the arguments the first instruction waits for them, and with it every launch behind
// (back to back, 1024 x 2048 at g = 32: 4.8 -> 5.4 us; 1 % on the median of the quantizer's launches).
template <bool HOLD>
__device__ __forceinline__ void pdl_begin() {
    if (!HOLD) pdl_launch_dependents();
    pdl_wait();
    if (HOLD) pdl_launch_dependents();
}

// 32 bytes in one access of a thread (both ends 32-byte aligned).  Threads that own 32 or 64 consecutive bytes touch whole
// sectors this way; with 16-byte accesses every sector is touched twice.
__device__ __forceinline__ void load32B(const void *p, uint32_t *w) {
    asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "l"(p));
}
__device__ __forceinline__ void store32B(void *p, const uint32_t *w) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}
__device__ __forceinline__ bool aligned32B(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 31) == 0; }
// N words (a multiple of 8) from or to a pointer that is only known to be 16-byte aligned.
template <int N>
__device__ __forceinline__ void load_words(const void *p, uint32_t (&w)[N]) {
    const uint8_t *b = reinterpret_cast<const uint8_t *>(p);
    if (aligned32B(p)) {
#pragma unroll
        for (int i = 0; i < N; i += 8) load32B(b + 4 * i, &w[i]);
    } else {
#pragma unroll
        for (int i = 0; i < N; i += 4) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(b + 4 * i));
            w[i] = v.x; w[i + 1] = v.y; w[i + 2] = v.z; w[i + 3] = v.w;
        }
    }
}
template <int N>
__device__ __forceinline__ void store_words(void *p, const uint32_t (&w)[N]) {
    uint8_t *b = reinterpret_cast<uint8_t *>(p);
    if (aligned32B(p)) {
#pragma unroll
        for (int i = 0; i < N; i += 8) store32B(b + 4 * i, &w[i]);
    } else {
#pragma unroll
        for (int i = 0; i < N; i += 4) *reinterpret_cast<uint4 *>(b + 4 * i) = make_uint4(w[i], w[i + 1], w[i + 2], w[i + 3]);
    }
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              int cluster_x, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    int n = 0;
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
    if (cluster_x > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)cluster_x;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = n;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
    return e == cudaSuccess ? cudaGetLastError() : e;
}
#endif

// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) applies to the current device only.  One static
// instance per kernel (per template instantiation of a launcher) remembers on which devices of this
// process the attribute has been set; setting it twice is harmless, so the race between two host
// threads that both see "not yet" is benign.
struct DynamicSmemOnce {
    bool done[64] = {};
    template <typename Kernel>
    cudaError_t set(Kernel kernel, int bytes) {
        int dev = -1;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
        return e;
    }
};

// Status / error plumbing.
int cuda_fail(cudaError_t e);             // records the message, returns QUEST_ERR_CUDA
int cuda_fail_msg(const char *msg);
int *device_status_word();                // device address of the timeout word (current device)
int check_device();                       // QUEST_OK iff current device is sm_10x
int num_sms();                            // of the current device

// Launchers (each returns a quest_status; arguments already validated).
// One tensor of a quantizer launch: rows of `x` -> any of codes / scales / mask / int8 GEMM
// operand / per-row sum of the operand bytes (each nullable).
struct QuantJob {
    const void *x;
    int64_t rows;
    int64_t ld;
    uint8_t *codes;
    float *scales;
    uint8_t *mask;
    int8_t *op8;
    int32_t *rowsum;
    uint16_t *rot = nullptr;   // [rows x cols] bfloat16 of the orthonormal rotation (no quantization needed for it)
    uint16_t *cbf = nullptr;   // [rows x cols] grid values as bfloat16
};
// Up to two tensors with the same row length, dtype and parameters share one launch.  for_decode: the launch
// precedes launch_decode.  That kernel may begin only once everything before the quantizer has finished (so that it
// may read, ahead of its own wait, what the quantizer does not write), and it takes x as signed bytes 2^(7-b) c at
// every width.
int launch_quantize(const QuantJob *jobs, int njobs, int dtype, int64_t cols, int bits, int had_block,
                    float trust_factor, cudaStream_t st, int grid = GRID_UNIFORM, bool for_decode = false);
// The inference layer with cached weights for a few rows of x, where decode_serves it (quest_decode.cu).  With w_codes the
// packed codes of w are the source and its operand (and row sums at 8 bits) is written to b8 / rs_b; otherwise b8
// holds it.  fused: x is quantized in the same launch (only if decode_fuses_quantizer), else by a launch_quantize
// for_decode directly before.
bool decode_serves(int64_t M, int64_t N, int64_t K, int bits, bool w_codes);
bool decode_fuses_quantizer(int64_t M, int64_t N, int64_t K);
int launch_decode(const QuantJob &jx, int dtype, bool fused, const uint8_t *wq, int8_t *b8, int32_t *rs_b, const float *sw,
                  bool w_codes, int64_t N, int64_t K, int bits, int had_block, float trust_factor, void *y, int y_dtype,
                  cudaStream_t st);
int launch_unpack(const uint8_t *codes, int bits, int64_t rows, int64_t K, int8_t *out,
                  int32_t *rowsum, cudaStream_t st, bool e2m1 = false);
// Packed codes -> tensor-core operands of one contraction in a single launch (an operand that is NULL is left out).
int launch_unpack_pair(const uint8_t *xq, int bits_x, int64_t M, int8_t *a8, const uint8_t *wq, int bits_w, int64_t N,
                       int8_t *b8, int64_t K, bool e2m1, cudaStream_t st);
// Row sums of two byte operands with the same row length, signed or unsigned, in one launch (NULL: not wanted).
int launch_rowsum_pair(const void *a, int64_t rows_a, bool unsigned_a, int32_t *out_a,
                       const void *b, int64_t rows_b, bool unsigned_b, int32_t *out_b, int64_t K, cudaStream_t st);
int launch_rowsum(const int8_t *a8, int64_t rows, int64_t K, int32_t *rowsum, cudaStream_t st);
int launch_gemm(const int8_t *a8, const int8_t *b8, const int32_t *rs_a, const int32_t *rs_b,
                int bits_x, int bits_w, const float *sx, const float *sw,
                int64_t M, int64_t N, int64_t K, void *y, int y_dtype, int64_t ldy,
                int32_t *acc, cudaStream_t st, bool x_codes = false, bool w_codes = false);   // *_codes: 8-bit codes as they are

int launch_gemm_swiglu(const int8_t *a8, const int8_t *b8, const int32_t *rs_a, const int32_t *rs_b, int bits,
                       const float *sx, const float *sw_gate, const float *sw_up, int64_t M, int64_t I, int64_t K,
                       void *h, cudaStream_t st);

int launch_bounded_wait_probe(long long limit_cycles, int *report, cudaStream_t st);

// Per-stage event timing (quest_stage_timing): bracket a stage of another translation unit.
void *stage_begin(int id, cudaStream_t st);
void stage_end(void *scope);

// opl: 1 a [I x Kc], b [Kc x J]; 2 a [Kc x I], b [Kc x J].
int launch_gemm_bf16_masked(const void *a, const void *b, int64_t I, int64_t J, int64_t Kc,
                            const uint8_t *mask, void *out, int out_dtype, int fuse_iht, int opl, cudaStream_t st);

// The same product in `parts` parts of the contraction index (divide_contraction says how many): bare binary32 sums, part q
// from row q * ((I + 255) / 256 * 256) of `out`.
int divide_contraction(int64_t I, int64_t J, int64_t Kc, int64_t rows_free, bool own_launch);
int launch_gemm_bf16_parts(const void *a, const void *b, int64_t I, int64_t J, int64_t Kc, float *out, int parts, int opl,
                           cudaStream_t st);

// Contraction of E2M1 nibble operands (tcgen05 kind::mxf4, unit block scales): acc = acc_mul * sum v_x v_w
// (int32, exact), y = sx sw sum v_x v_w.  xq, wq 16-byte aligned, K % 32 == 0.  Serves the FP4 grid
// (acc_mul = 4) and, inside launch_gemm, the one- and two-bit uniform grids (acc_mul = 1).
int launch_gemm_e2m1(const uint8_t *xq, const uint8_t *wq, const float *sx, const float *sw, int64_t M, int64_t N,
                     int64_t K, void *y, int y_dtype, int64_t ldy, int32_t *acc, int acc_mul, cudaStream_t st);
// Weight-only contraction: y[m][n] = sw[n] * sum_k a[m][k] b[n][k], bfloat16 operands (dense, K contiguous),
// binary32 accumulation.
int launch_gemm_bf16_scaled(const void *a, const void *b, const float *sw, int64_t M, int64_t N, int64_t K,
                            void *y, int y_dtype, int64_t ldy, cudaStream_t st);

}  // namespace quest
