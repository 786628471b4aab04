// wm_backward.cu -- wm_mdn_nll_backward: the world model's training step, the gradient
// of the teacher-forced mixture NLL (Sec. 4.7) by backpropagation through time
// (Sec. 3.3.2).
//
// Rows are (step, sequence) pairs r = t N + n, time-major like every [T, N, ...] array of
// the library.  Everything that does not depend on the recurrence is batched over all
// N T rows:
//   forward      the teacher-forced pass of the kernel family wm_mdn_nll picks, keeping
//                h_t and c_t of every row
//   X, Y         the GEMM operands of every row, X = [op(z_t); op(h_{t-1})], Y = op(h_t): the
//                forward's own operand rows where it leaves them, else built (k_bw_build)
//   gates        the pre-activations G = X W_zh + b + W_a[a_t]: left by the forward's one-launch
//                recurrence, else one GEMM and, with sigma / tanh, k_bw_gates
//   dMD          d NLL / d [logit | mu | log sigma] of every counted row: formed by the
//                tensor family's head GEMM, else from the head outputs          (k_bw_mdn)
//   dY           dMD W_mdn^T (one GEMM): the heads' share of d loss / d h_t
// then the recurrence, t = T-1 .. 0, in one launch (wm_brecur.cu) or per step:
//   dG_t         the cell's backward step from dY_t + dH and the carried dc  (k_bw_cell)
//   dH           dG_t W_h^T (one GEMM on N rows): d loss / d h_{t-1}
// and the weight gradients, batched again:
//   dW_z, dW_h   X^T dG (two GEMMs writing the z and h rows of the output)
//   dW_a         per action, the sum of the dG rows that took it          (k_bw_arows)
//   dW_mdn       Y^T dMD (one GEMM)
//   db_lstm      the sum of dW_a's buckets, one of them for rows without an action
//   db_mdn       column sums                                               (k_bw_colsum4)
// The plain GEMMs are cuBLAS calls (bf16 operands and fp32 accumulation on the bf16 path;
// on the fp32 path the library's fp32 emulation, and for the recurrence's dH bf16 products
// of the operands' hi and lo parts, see k_bw_split3); the rest are the kernels below.
// Every reduction has a fixed order, so results are bit-reproducible.
#include <cublas_v2.h>
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>

#include "wm_internal.h"

namespace {

constexpr int CHUNKS = 16;  // row chunks of the two-level reductions

template <class T> __device__ __forceinline__ T to_op(float v);
template <> __device__ __forceinline__ float to_op<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 to_op<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// X [NT, Z+H] = [z_t | h_{t-1}] and Y [NT, H] = h_t, in the GEMM operand type (bf16: RNE,
// the forward's operand rounding)
// (a block per row at a time, the row's columns over its threads: no 64-bit divisions)
template <class T>
__global__ void k_bw_build(int N, int TT, int Z, int H, const float *__restrict__ z_seq,
                           const float *__restrict__ hs, T *__restrict__ X, T *__restrict__ Y) {
    const int KX = Z + H;
    const size_t NT = (size_t)N * TT;
    for (size_t r = blockIdx.x; r < NT; r += gridDim.x) {
        const float *hp = r >= (size_t)N ? hs + (r - N) * H : nullptr;  // h_{-1} = 0
        for (int k = threadIdx.x; k < KX; k += blockDim.x) {
            const float v = k < Z ? z_seq[r * Z + k] : (hp ? hp[k - Z] : 0.f);
            X[r * KX + k] = to_op<T>(v);
        }
        for (int k = threadIdx.x; k < H; k += blockDim.x) Y[r * H + k] = to_op<T>(hs[r * H + k]);
    }
}

// gate pre-activations + bias + the action row -> i, f, g, o (in place); a block per row at
// a time, four columns per thread
__global__ void k_bw_gates(size_t NT, int N, int H, int A, float *__restrict__ G, const int32_t *__restrict__ act,
                           const float *__restrict__ Wa, const float *__restrict__ bias) {
    const int H4 = 4 * H;
    for (size_t r = blockIdx.x; r < NT; r += gridDim.x) {
        const int a = act[r];
        const float *wa = (a >= 0 && a < A) ? Wa + (size_t)a * H4 : nullptr;
        float4 *g4 = reinterpret_cast<float4 *>(G + r * H4);
        for (int c4 = threadIdx.x; c4 < H4 / 4; c4 += blockDim.x) {
            const int col = 4 * c4;
            float4 v = g4[c4];
            float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float u = x[j] + bias[col + j];
                if (wa) u += wa[col + j];
                const bool cand = col + j >= 2 * H && col + j < 3 * H;  // the g gate: tanh
                x[j] = cand ? tanhf(u) : 1.f / (1.f + expf(-u));
            }
            g4[c4] = make_float4(x[0], x[1], x[2], x[3]);
        }
    }
}

// d NLL / d [logit | mu | log sigma] of one row's latent dim d (0 past the row's length)
// (where the forward's head GEMM did not form it)
__global__ void k_bw_mdn(int N, int TT, int Z, int K, const float *__restrict__ md, const float *__restrict__ z_seq,
                         const int32_t *__restrict__ lengths, float *__restrict__ dmd, __nv_bfloat16 *__restrict__ dmd_op) {
    const int KZ = K * Z, M = 3 * KZ;
    const size_t NT = (size_t)N * TT;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < NT * Z; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / Z;
        const int d = (int)(i % Z), t = (int)(r / N), n = (int)(r % N);
        int len = lengths ? lengths[n] : TT;
        len = len < 0 ? 0 : (len > TT ? TT : len);
        const float *row = md + r * M;
        float *out = dmd + r * M;
        __nv_bfloat16 *oop = dmd_op ? dmd_op + r * M : nullptr;  // bf16 path: the GEMMs' operand
        if (t >= len) {
            for (int k = 0; k < K; ++k)
                for (int p = 0; p < 3; ++p) {
                    out[p * KZ + d * K + k] = 0.f;
                    if (oop) oop[p * KZ + d * K + k] = __float2bfloat16_rn(0.f);
                }
            continue;
        }
        const float x = z_seq[(r + N) * Z + d];  // the target z_{t+1}
        const float *lg = row + d * K, *mu = row + KZ + d * K, *ls = row + 2 * KZ + d * K;
        float lmax = -INFINITY, s = 0.f, term[32], tmax = -INFINITY, acc = 0.f;
        for (int k = 0; k < K; ++k) lmax = fmaxf(lmax, lg[k]);
        for (int k = 0; k < K; ++k) s += expf(lg[k] - lmax);
        const float logz = lmax + logf(s);
        for (int k = 0; k < K; ++k) {
            const float zs = (x - mu[k]) * expf(-ls[k]);
            term[k] = (lg[k] - logz) - 0.5f * zs * zs - ls[k] - 0.91893853320467274178f;
            tmax = fmaxf(tmax, term[k]);
        }
        for (int k = 0; k < K; ++k) acc += expf(term[k] - tmax);
        const float lse = tmax + logf(acc);
        for (int k = 0; k < K; ++k) {
            const float pi = expf(lg[k] - logz), gam = expf(term[k] - lse);
            const float is = expf(-ls[k]), zs = (x - mu[k]) * is;
            const float v0 = pi - gam, v1 = -gam * zs * is, v2 = gam * (1.f - zs * zs);
            out[d * K + k] = v0;
            out[KZ + d * K + k] = v1;
            out[2 * KZ + d * K + k] = v2;
            if (!oop) continue;
            oop[d * K + k] = __float2bfloat16_rn(v0);
            oop[KZ + d * K + k] = __float2bfloat16_rn(v1);
            oop[2 * KZ + d * K + k] = __float2bfloat16_rn(v2);
        }
    }
}

// The cell's backward step at t for N rows: dh = dY_t + dH (from step t + 1), and
//   dc = dh o (1 - tanh^2 c_t) + dc_carried;  dG = [dc g i(1-i) | dc c_{t-1} f(1-f) |
//   dc i (1-g^2) | dh tanh(c_t) o(1-o)];  dc_carried <- dc f.
__global__ void k_bw_cell(int N, int H, int t, int first, const float *__restrict__ act, const float *__restrict__ cs,
                          const float *__restrict__ dY, const float *__restrict__ dH, float *__restrict__ dC,
                          float *__restrict__ dG, __nv_bfloat16 *__restrict__ dG_op, __nv_bfloat16 *__restrict__ dG3) {
    const size_t base = (size_t)t * N;
    const int u = blockIdx.x * blockDim.x + threadIdx.x;  // unit; rows n over the grid's y
    if (u >= H) return;
    for (size_t n = blockIdx.y; n < (size_t)N; n += gridDim.y) {
        const size_t i = n * H + u;
        const size_t r = base + n;
        const float *a = act + r * 4 * H;
        const float ig = a[u], fg = a[H + u], gg = a[2 * H + u], og = a[3 * H + u];
        const float c = cs[r * H + u], cp = t > 0 ? cs[(r - N) * H + u] : 0.f;
        const float dh = dY[r * H + u] + (first ? 0.f : dH[i]);
        const float tc = tanhf(c);
        const float dc = dh * og * (1.f - tc * tc) + (first ? 0.f : dC[i]);
        const float g0 = dc * gg * ig * (1.f - ig), g1 = dc * cp * fg * (1.f - fg);
        const float g2 = dc * ig * (1.f - gg * gg), g3 = dh * tc * og * (1.f - og);
        float *o = dG + r * 4 * H;
        o[u] = g0; o[H + u] = g1; o[2 * H + u] = g2; o[3 * H + u] = g3;
        if (dG_op) {  // bf16 path: the GEMMs' operand
            __nv_bfloat16 *oo = dG_op + r * 4 * H;
            oo[u] = __float2bfloat16_rn(g0); oo[H + u] = __float2bfloat16_rn(g1);
            oo[2 * H + u] = __float2bfloat16_rn(g2); oo[3 * H + u] = __float2bfloat16_rn(g3);
        }
        if (dG3) {  // this step's row as [hi | hi | lo] for the three-product recurrence GEMM
            __nv_bfloat16 *q = dG3 + n * 12 * H;
            const float gv[4] = {g0, g1, g2, g3};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const __nv_bfloat16 hi = __float2bfloat16_rn(gv[j]);
                q[j * H + u] = hi;
                q[4 * H + j * H + u] = hi;
                q[8 * H + j * H + u] = __float2bfloat16_rn(gv[j] - __bfloat162float(hi));
            }
        }
        dC[i] = dc * fg;
    }
}

// Compensated (Kahan) fp32 sum: the error stays near one rounding however many terms.
struct Kahan {
    float s = 0.f, comp = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float y = v - comp, t = s + y;
        comp = (t - s) - y;
        s = t;
    }
};

// Column sums of a [R, C] matrix, two levels: chunk c of the rows (COLSUM_CHUNKS of them)
// into part[c][C], then the chunks' partials in order.  The order, so the result, is fixed.
// C % 4 == 0: a thread takes four columns and every fourth row of the chunk, and the four row
// lanes are combined in order (one column a thread and all rows: 106 us for 65,536 x 960, bound by
// the loads in flight).  Other C: one thread per column, rows in order.
constexpr int COLSUM_CHUNKS = 64;
__global__ void __launch_bounds__(256) k_bw_colsum4(size_t R, int C, const float *__restrict__ in, float *__restrict__ part) {
    __shared__ float4 lanes[3][64];
    const int q = threadIdx.x & 63, l = threadIdx.x >> 6, col = 4 * (blockIdx.x * 64 + q), c = blockIdx.y;
    const size_t r0 = R * c / COLSUM_CHUNKS, r1 = R * (c + 1) / COLSUM_CHUNKS;
    Kahan k[4];
    if (col < C) {
#pragma unroll 8
        for (size_t r = r0 + l; r < r1; r += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(in + r * C + col);
            k[0].add(v.x); k[1].add(v.y); k[2].add(v.z); k[3].add(v.w);
        }
    }
    if (l) lanes[l - 1][q] = make_float4(k[0].s, k[1].s, k[2].s, k[3].s);
    __syncthreads();
    if (l || col >= C) return;
    for (int i = 0; i < 3; ++i) {
        const float4 v = lanes[i][q];
        k[0].add(v.x); k[1].add(v.y); k[2].add(v.z); k[3].add(v.w);
    }
    *reinterpret_cast<float4 *>(part + (size_t)c * C + col) = make_float4(k[0].s, k[1].s, k[2].s, k[3].s);
}
__global__ void k_bw_colsum(size_t R, int C, const float *__restrict__ in, float *__restrict__ part) {
    const int col = blockIdx.x * blockDim.x + threadIdx.x, c = blockIdx.y;
    if (col >= C) return;
    const size_t r0 = R * c / COLSUM_CHUNKS, r1 = R * (c + 1) / COLSUM_CHUNKS;
    Kahan k;
    for (size_t r = r0; r < r1; ++r) k.add(in[r * C + col]);
    part[(size_t)c * C + col] = k.s;
}
__global__ void k_bw_colsum_fin(int C, const float *__restrict__ part, float *__restrict__ out) {
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= C) return;
    double s = 0.0;
    for (int c = 0; c < COLSUM_CHUNKS; ++c) s += part[(size_t)c * C + col];
    out[col] = (float)s;
}

// The action rows of dW_lstm: dW_a[a] = sum of the dG rows whose action is a, and bucket A the rows
// without an action.  Each row chunk is first sorted stably by bucket (k_bw_rowsort: one block per
// chunk, rows taken in order by one warp 32 at a time, each lane's place among the lanes with the same
// bucket from a match mask), then block (a, c) sums, in row order, only the rows of chunk c in bucket a,
// into part[c][a][4H]; then the CHUNKS partials in order.  db_lstm is the sum of all buckets'
// partials: dG (fp32, half a gigabyte at 65,536 rows of H = 512) is read once for both.
__global__ void k_bw_rowsort(size_t R, int A, const int32_t *__restrict__ act, int32_t *__restrict__ srows,
                             int32_t *__restrict__ soff) {
    extern __shared__ int s_cnt[];  // [A + 1] counts, then running cursors
    const int c = blockIdx.x;
    const size_t r0 = R * c / CHUNKS, r1 = R * (c + 1) / CHUNKS;
    for (int a = threadIdx.x; a <= A; a += blockDim.x) s_cnt[a] = 0;
    __syncthreads();
    for (size_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) {
        const int a = act[r];
        atomicAdd(&s_cnt[a >= 0 && a < A ? a : A], 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {  // exclusive offsets within the chunk
        int run = 0;
        int32_t *off = soff + (size_t)c * (A + 2);
        for (int a = 0; a <= A; ++a) {
            const int n = s_cnt[a];
            off[a] = run;
            s_cnt[a] = run;
            run += n;
        }
        off[A + 1] = run;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        for (size_t b8 = r0; b8 < r1; b8 += 256) {  // eight loads in flight, then their rows in order
            int av[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const size_t r = b8 + 32 * i + lane;
                av[i] = r < r1 ? act[r] : -1;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const size_t r = b8 + 32 * i + lane;
                const bool ok = r < r1;
                const int a = ok && (av[i] < 0 || av[i] >= A) ? A : av[i];
                const uint32_t same = __match_any_sync(0xffffffffu, a);
                const int rank = __popc(same & ((1u << lane) - 1u));
                int pos = 0;
                if (ok) pos = s_cnt[a] + rank;
                __syncwarp();
                if (ok && rank == 0) s_cnt[a] += __popc(same);  // the lowest lane of each action
                __syncwarp();
                if (ok) srows[r0 + pos] = (int32_t)r;
            }
        }
    }
}
__global__ void __launch_bounds__(256) k_bw_arows(size_t R, int A, int H4, const int32_t *__restrict__ srows,
                                                  const int32_t *__restrict__ soff, const float *__restrict__ dG,
                                                  float *__restrict__ part) {
    const int a = blockIdx.x, c = blockIdx.y;
    const size_t r0 = R * c / CHUNKS;
    const int32_t *off = soff + (size_t)c * (A + 2);
    const int i0 = off[a], i1 = off[a + 1];
    for (int col = 4 * threadIdx.x; col < H4; col += 4 * blockDim.x) {  // (H4 is a multiple of 4)
        Kahan k[4];
#pragma unroll 8
        for (int i = i0; i < i1; ++i) {
            const float4 v = *reinterpret_cast<const float4 *>(dG + (size_t)srows[r0 + i] * H4 + col);
            k[0].add(v.x); k[1].add(v.y); k[2].add(v.z); k[3].add(v.w);
        }
        *reinterpret_cast<float4 *>(part + ((size_t)c * (A + 1) + a) * H4 + col) = make_float4(k[0].s, k[1].s, k[2].s, k[3].s);
    }
}
__global__ void k_bw_arows_fin(int A, int H4, const float *__restrict__ part, float *__restrict__ out) {
    const size_t n = (size_t)A * H4, ld = (size_t)(A + 1) * H4;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        float s = 0.f;
#pragma unroll
        for (int c = 0; c < CHUNKS; ++c) s += part[(size_t)c * ld + i];
        out[i] = s;
    }
}

// bf16 copies of the weights the backward's GEMMs read (bf16 path): W_zh [Z+H, 4H] and
// W_mdn [H, M] from the stepwise family's (already bf16-rounded) fp32 matrices
__global__ void k_bw_cast(size_t rows, int cols, const float *__restrict__ src, long lds, __nv_bfloat16 *__restrict__ dst) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < rows * cols; i += (size_t)gridDim.x * blockDim.x)
        dst[i] = __float2bfloat16_rn(src[(i / cols) * lds + i % cols]);
}

// W_h [H, 4H] (the h rows of the gate matrix) as bf16 rows [hi | lo | hi], hi = bf16(w),
// lo = bf16(w - hi): against a [hi | hi | lo] row of dG the K = 12H contraction is
// hi.hi + hi.lo + lo.hi, the fp32 product up to the dropped lo.lo term and the parts'
// residuals (at most about 3 * 2^-16 of each product: bf16's unit roundoff is 2^-8)
__global__ void k_bw_split3(size_t rows, int cols, const float *__restrict__ src, long lds,
                            __nv_bfloat16 *__restrict__ dst) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < rows * cols; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / cols;
        const int k = (int)(i % cols);
        const float w = src[r * lds + k];
        const __nv_bfloat16 hi = __float2bfloat16_rn(w), lo = __float2bfloat16_rn(w - __bfloat162float(hi));
        __nv_bfloat16 *d = dst + r * 3 * cols;
        d[k] = hi;
        d[cols + k] = lo;
        d[2 * cols + k] = hi;
    }
}

int grid_of(size_t n) {
    size_t g = (n + 255) / 256;
    if (g > 8192) g = 8192;
    return g < 1 ? 1 : (int)g;
}

inline size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

// Row-major GEMM on cuBLAS: C[m][n] = sum_k A(m,k) B(k,n), A(m,k) = ta ? A[k lda + m] :
// A[m lda + k], B(k,n) = tb ? B[n ldb + k] : B[k ldb + n].  (cuBLAS is column-major: it
// computes C^T = B^T A^T.)  bf16 operands accumulate in fp32; fp32 operands take cuBLAS's
// fp32 emulation on the tensor cores (each operand split into three bf16 parts, fp32-accurate
// products), or plain fp32 where the library does not offer it.
cublasStatus_t gemm(cublasHandle_t hb, bool bf16, bool ta, bool tb, int m, int n, int k, const void *A, long lda,
                    const void *B, long ldb, float *C, long ldc, float beta = 0.f) {
    const float one = 1.f;
    const cudaDataType_t dt = bf16 ? CUDA_R_16BF : CUDA_R_32F;
    auto run = [&](cublasComputeType_t ct) {
        return cublasGemmEx(hb, tb ? CUBLAS_OP_T : CUBLAS_OP_N, ta ? CUBLAS_OP_T : CUBLAS_OP_N, n, m, k, &one, B, dt,
                            (int)ldb, A, dt, (int)lda, &beta, C, CUDA_R_32F, (int)ldc, ct, CUBLAS_GEMM_DEFAULT);
    };
    if (bf16) return run(CUBLAS_COMPUTE_32F);
    const cublasStatus_t st = run(CUBLAS_COMPUTE_32F_EMULATED_16BFX9);
    return st == CUBLAS_STATUS_NOT_SUPPORTED ? run(CUBLAS_COMPUTE_32F_PEDANTIC) : st;
}

cudaError_t cublas_err(cublasStatus_t st) {
    return st == CUBLAS_STATUS_SUCCESS ? cudaSuccess
                                       : st == CUBLAS_STATUS_ALLOC_FAILED ? cudaErrorMemoryAllocation
                                                                          : cudaErrorUnknown;
}

}  // namespace

// X and Y are built unless the forward left them: its operand rows (bf16; h_t is then read from them
// alone), or z_seq and h_t as they are (fp32, when no product with W_zh is left to do: h_{t-1} is
// then h_t's row N rows up).  Head outputs are kept unless the forward formed their gradient.
wm_bw_fwd wm_bw_plan(const wm_handle *h, int N, int T, bool tensor) {
    const bool bf = h->cfg.precision == WM_BF16;
    wm_bw_fwd f{};
    wm_brecur_args a{};
    f.have_dmd = tensor;
    f.have_g = tensor && T > 1 && (size_t)N * T < (1u << 30) && wm_tc_scores_in_one(h, N, T) &&
               wm_brecur_plan(h, N, h->cfg.h_dim, &a);  // (the backward recurrence reads pre-activations)
    f.built = bf ? !tensor : !f.have_g;
    return f;
}

// The forward's outputs at the front of the backward's workspace, then its own buffers.
void wm_bw_carve(const wm_handle *h, int N, int T, void *base, wm_bw_fwd *f, void **tail) {
    const size_t NT = (size_t)N * T, H = h->cfg.h_dim, M = h->M;
    char *p = (char *)base;
    if (f->built || h->cfg.precision == WM_FP32) { f->hs = (float *)p; p += al(NT * H * 4); }
    f->cs = (float *)p; p += al(NT * H * 4);
    if (!f->have_dmd) { f->md = (float *)p; p += al(NT * M * 4); }
    f->nll = (float *)p; p += al((size_t)N * 4);
    f->G = (float *)p; p += al(NT * 4 * H * 4);
    f->dMD = (float *)p; p += al(NT * M * 4);
    f->dMDo = nullptr;
    if (h->cfg.precision == WM_BF16) { f->dMDo = (__nv_bfloat16 *)p; p += al(NT * M * 2); }
    *tail = p;
}

size_t wm_bw_ws(const wm_handle *h, int N, int T, const wm_bw_fwd &f) {
    const wm_config &c = h->cfg;
    const size_t Z = c.z_dim, A = c.a_dim, H = c.h_dim, M = h->M, KX = Z + H, H4 = 4 * H;
    const size_t NT = (size_t)N * T, es = c.precision == WM_BF16 ? 2 : 4;
    const size_t part_cols = H4 > M ? H4 : M;
    return (f.built || es == 4 ? al(NT * H * 4) : 0) + al(NT * H * 4)          // h, c
           + (f.have_dmd ? 0 : al(NT * M * 4)) + al((size_t)N * 4)             // head outputs, nll
           + (f.built ? al(NT * KX * es) + al(NT * H * es) : 0)                // X, Y
           + al(NT * H4 * 4)                                                   // gate activations
           + al(NT * M * 4) + (es == 2 ? al(NT * M * 2) : 0)                   // dMD
           + al(NT * H * 4)                                                    // dY
           + al(NT * H4 * 4) + (es == 2 ? al(NT * H4 * 2) : 0)                 // dG
           + 2 * al((size_t)N * H * 4)                                         // dH, dc
           + al((size_t)COLSUM_CHUNKS * part_cols * 4) + al((size_t)CHUNKS * (A + 1) * H4 * 4)  // partials
           + al(NT * 4) + al((size_t)CHUNKS * (A + 2) * 4)                       // rows sorted by action
           + (es == 4 ? al((size_t)N * 4 * H4 * 2) : 0)                          // fp32: dG_t as bf16 parts
           + al((size_t)(N / 128 + 1) * 4) + 256;                                // row-tile counters
}

cudaError_t wm_bw_prepare(wm_handle *h) {
    const cudaError_t re = wm_brecur_prepare(h);
    if (re != cudaSuccess) return re;
    if (!h->cublas) {
        cublasHandle_t hb;
        cublasStatus_t st = cublasCreate(&hb);
        if (st != CUBLAS_STATUS_SUCCESS) return cublas_err(st);
        h->cublas = hb;
        // fp32 GEMMs: the emulation whenever the library has it, and without the scans and
        // patches for infinities and NaNs (every operand here is finite: activations, their
        // gradients and the weights); where the library lacks either setting, its default
        cublasSetEmulationStrategy(hb, CUBLAS_EMULATION_STRATEGY_EAGER);
        cublasSetEmulationSpecialValuesSupport(hb, CUDA_EMULATION_SPECIAL_VALUES_SUPPORT_NONE);
    }
    const wm_config &c = h->cfg;
    if (c.precision == WM_BF16 && !h->bw_wzh) {
        const size_t Z = c.z_dim, A = c.a_dim, H = c.h_dim, M = h->M, KX = Z + H;
        cudaError_t e = cudaMalloc(&h->bw_wzh, KX * 4 * H * 2);
        if (e == cudaSuccess) e = cudaMalloc(&h->bw_wm, H * M * 2);
        if (e != cudaSuccess) return e;
        k_bw_cast<<<grid_of(KX * 4 * H), 256>>>(KX, 4 * (int)H, h->step.Wg, (long)(4 * H + A), (__nv_bfloat16 *)h->bw_wzh);
        k_bw_cast<<<grid_of(H * M), 256>>>(H, (int)M, h->step.Wh, (long)(M + h->NR), (__nv_bfloat16 *)h->bw_wm);
        e = cudaDeviceSynchronize();
        if (e != cudaSuccess) return e;
    }
    if (c.precision != WM_BF16 && !h->bw_w3) {
        const size_t Z = c.z_dim, A = c.a_dim, H = c.h_dim;
        cudaError_t e = cudaMalloc(&h->bw_w3, H * 12 * H * 2);
        if (e != cudaSuccess) return e;
        k_bw_split3<<<grid_of(H * 4 * H), 256>>>(H, 4 * (int)H, h->step.Wg + Z * (4 * H + A), (long)(4 * H + A),
                                                 (__nv_bfloat16 *)h->bw_w3);
        e = cudaDeviceSynchronize();
        if (e != cudaSuccess) return e;
    }
    if (c.precision != WM_BF16 && !h->bw_wm) {
        // W_mdn without the reward and done columns: the step layout's row stride M + NR is not a
        // multiple of 16 bytes, which keeps cuBLAS off the tensor cores for dY = dMD W_mdn^T
        const size_t H = c.h_dim, M = h->M;
        cudaError_t e = cudaMalloc(&h->bw_wm, H * M * 4);
        if (e == cudaSuccess)
            e = cudaMemcpy2D(h->bw_wm, M * 4, h->step.Wh, (M + h->NR) * 4, M * 4, H, cudaMemcpyDeviceToDevice);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

void wm_bw_free(wm_handle *h) {
    if (h->cublas) cublasDestroy((cublasHandle_t)h->cublas);
    cudaFree(h->bw_wzh);
    cudaFree(h->bw_wm);
    cudaFree(h->bw_w3);
    cudaFree(h->bws);
    h->cublas = h->bw_wzh = h->bw_wm = h->bw_w3 = h->bws = nullptr;
    h->bws_bytes = 0;
}

template <class T>
static cudaError_t bw_run(const wm_handle *h, int N, int TT, const float *z_seq, const int32_t *actions,
                          const int32_t *lengths, const wm_grads &g, const wm_bw_fwd &f, char *p, cudaStream_t s) {
    const wm_config &c = h->cfg;
    const bool bf = c.precision == WM_BF16;
    const int Z = c.z_dim, A = c.a_dim, H = c.h_dim, M = h->M, KX = Z + H, H4 = 4 * H;
    const size_t NT = (size_t)N * TT;
    cublasHandle_t hb = (cublasHandle_t)h->cublas;
    cublasStatus_t st = cublasSetStream(hb, s);
    if (st != CUBLAS_STATUS_SUCCESS) return cublas_err(st);
    const float *hs = f.hs, *cs = f.cs;
    float *G = f.G;
    const bool built = f.built;
    T *X = (T *)p;
    if (built) p += al(NT * KX * sizeof(T));
    T *Y = (T *)p;
    if (built) p += al(NT * H * sizeof(T));
    float *dMD = f.dMD;
    const void *dMDo = bf ? (const void *)f.dMDo : (const void *)dMD;  // the GEMMs' operand
    float *dY = (float *)p; p += al(NT * H * 4);
    float *dG = (float *)p; p += al(NT * H4 * 4);
    __nv_bfloat16 *dGo = bf ? (__nv_bfloat16 *)p : nullptr;  // bf16 path: dG as the GEMMs' operand
    if (bf) p += al(NT * H4 * 2);
    float *dH = (float *)p; p += al((size_t)N * H * 4);
    float *dC = (float *)p; p += al((size_t)N * H * 4);
    float *part = (float *)p; p += al((size_t)COLSUM_CHUNKS * (H4 > M ? H4 : M) * 4);
    float *apart = (float *)p; p += al((size_t)CHUNKS * (A + 1) * H4 * 4);
    int32_t *srows = (int32_t *)p; p += al(NT * 4);
    int32_t *soff = (int32_t *)p; p += al((size_t)CHUNKS * (A + 2) * 4);
    // fp32: dG_t as [hi | hi | lo], or, in the one-launch recurrence, two steps' rows [hi | lo]
    __nv_bfloat16 *dG3 = bf ? nullptr : (__nv_bfloat16 *)p;
    if (!bf) p += al((size_t)N * 4 * H4 * 2);
    int *count = (int *)p;
    // weights of the GEMMs: W_zh = the z and h rows of the gate matrix, W_mdn, W_h = W_zh's h rows
    const void *Wzh = bf ? (const void *)h->bw_wzh : (const void *)h->step.Wg;
    const long ldw = bf ? H4 : H4 + A;
    const void *Wm = h->bw_wm;
    const long ldm = M;
    const void *Wh = bf ? (const void *)((const __nv_bfloat16 *)h->bw_wzh + (size_t)Z * H4)
                        : (const void *)(h->step.Wg + (size_t)Z * (H4 + A));
    int launches = 0;
    if (built) {
        wm_ktime kt(h, WM_KERNEL_BW, s);
        k_bw_build<T><<<(unsigned)(NT < 8192 ? NT : 8192), 256, 0, s>>>(N, TT, Z, H, z_seq, hs, X, Y);
        ++launches;
    }
    const void *Xz = built ? (const void *)X : bf ? (const void *)f.frames : (const void *)z_seq;
    const long ldx = built ? KX : bf ? f.ld : Z;
    if (!f.have_g) {
        wm_ktime kt(h, WM_KERNEL_BW_GEMM, s);
        if (built) {
            st = gemm(hb, bf, false, false, (int)NT, H4, KX, X, KX, Wzh, ldw, G, H4);
        } else {  // z columns, then h columns on top (the rows' padding between them is skipped)
            st = gemm(hb, true, false, false, (int)NT, H4, Z, f.frames, f.ld, Wzh, ldw, G, H4);
            if (st == CUBLAS_STATUS_SUCCESS)
                st = gemm(hb, true, false, false, (int)NT, H4, H, f.frames + f.h_col, f.ld,
                          (const __nv_bfloat16 *)h->bw_wzh + (size_t)Z * H4, ldw, G, H4, 1.f);
            ++launches;
        }
        ++launches;
    }
    if (st != CUBLAS_STATUS_SUCCESS) return cublas_err(st);
    if (!f.have_g || !f.have_dmd) {
        wm_ktime kt(h, WM_KERNEL_BW, s);
        if (!f.have_g)
            k_bw_gates<<<(unsigned)(NT < 8192 ? NT : 8192), 256, 0, s>>>(NT, N, H, A, G, actions, h->step.Wa, h->step.bg);
        if (!f.have_dmd) k_bw_mdn<<<grid_of(NT * Z), 256, 0, s>>>(N, TT, Z, c.k_mix, f.md, z_seq, lengths, dMD, f.dMDo);
        launches += !f.have_g + !f.have_dmd;
    }
    {
        wm_ktime kt(h, WM_KERNEL_BW_GEMM, s);
        st = gemm(hb, bf, false, true, (int)NT, H, M, dMDo, M, Wm, ldm, dY, H);
        ++launches;
    }
    if (st != CUBLAS_STATUS_SUCCESS) return cublas_err(st);
    wm_brecur_args ra{};
    const bool one = TT > 1 && NT < (1u << 30) && wm_brecur_plan(h, N, H, &ra);
    if (one) {
        CUtensorMap gm, wmap;
        // (bw_wzh: rows z | h of 4H columns; bw_w3: rows [hi | lo | hi])
        if (!(bf ? wm_tc_make_map(&gm, dGo, NT, H4, 128) && wm_tc_make_map(&wmap, h->bw_wzh, KX, H4, 64)
                 : wm_tc_make_map(&gm, dG3, 2 * (size_t)N, 2 * H4, 128) && wm_tc_make_map(&wmap, h->bw_w3, H, 3 * H4, 64)))
            return cudaErrorInvalidValue;
        ra.N = N; ra.T = TT; ra.H = H;
        ra.act = G; ra.cs = cs; ra.dY = dY; ra.pre = f.have_g;
        ra.dG = dG; ra.dGo = dGo; ra.parts = dG3;
        ra.count = count; ra.status = h->status; ra.w_row0 = bf ? Z : 0;
        ra.test_wait = h->test_wait;  // an injected wait that the forward did not take
        h->test_wait = 0;
        cudaError_t e = cudaMemsetAsync(count, 0, (size_t)ra.m_tiles * 4, s);
        if (e != cudaSuccess) return e;
        wm_ktime kt(h, WM_KERNEL_BW, s);
        if ((e = wm_brecur_launch(!bf, &gm, &wmap, ra, s)) != cudaSuccess) return e;
        launches += (ra.m_tiles + ra.m_per_launch - 1) / ra.m_per_launch;
    }
    for (int t = TT - 1; t >= 0 && !one; --t) {
        {
            wm_ktime kt(h, WM_KERNEL_BW, s);
            const dim3 grid((unsigned)((H + 255) / 256), (unsigned)(N < 65535 ? N : 65535));
            k_bw_cell<<<grid, 256, 0, s>>>(N, H, t, t == TT - 1, G, cs, dY, dH, dC, dG, dGo, t > 0 ? dG3 : nullptr);
            ++launches;
        }
        if (t > 0) {
            wm_ktime kt(h, WM_KERNEL_BW_GEMM, s);
            // fp32: bf16 operands over K = 12H (three products, fp32 accumulation)
            st = bf ? gemm(hb, true, false, true, N, H, H4, dGo + (size_t)t * N * H4, H4, Wh, ldw, dH, H)
                    : gemm(hb, true, false, true, N, H, 3 * H4, dG3, 3 * H4, h->bw_w3, 3 * H4, dH, H);
            ++launches;
            if (st != CUBLAS_STATUS_SUCCESS) return cublas_err(st);
        }
    }
    {
        wm_ktime kt(h, WM_KERNEL_BW_GEMM, s);
        // z rows and h rows of dW_lstm: X^T dG, straight into the output's row blocks
        const void *dGx = bf ? (const void *)dGo : (const void *)dG;  // fp32: dG itself
        st = gemm(hb, bf, true, false, Z, H4, (int)NT, Xz, ldx, dGx, H4, g.W_lstm, H4);
        float *dWh = g.W_lstm + (size_t)(Z + A) * H4;
        if (st == CUBLAS_STATUS_SUCCESS)
            st = built ? gemm(hb, bf, true, false, H, H4, (int)NT, X + Z, KX, dGx, H4, dWh, H4)
                 : bf  ? gemm(hb, true, true, false, H, H4, (int)NT, f.frames + f.h_col, f.ld, dGx, H4, dWh, H4)
                       : gemm(hb, false, true, false, H, H4, (int)(NT - N), hs, H, dG + (size_t)N * H4, H4, dWh, H4);
        const void *Yx = built ? (const void *)Y : bf ? (const void *)(f.frames + (size_t)N * f.ld + f.h_col) : (const void *)hs;
        if (st == CUBLAS_STATUS_SUCCESS)
            st = gemm(hb, bf, true, false, H, M, (int)NT, Yx, built || !bf ? H : f.ld, dMDo, M, g.W_mdn, M);
        launches += 3;
    }
    if (st != CUBLAS_STATUS_SUCCESS) return cublas_err(st);
    {
        wm_ktime kt(h, WM_KERNEL_BW, s);
        auto colsum = [&](size_t R, int C, const float *in, float *out) {
            if (C % 4 == 0) k_bw_colsum4<<<dim3((C + 255) / 256, COLSUM_CHUNKS), 256, 0, s>>>(R, C, in, part);
            else k_bw_colsum<<<dim3((C + 255) / 256, COLSUM_CHUNKS), 256, 0, s>>>(R, C, in, part);
            k_bw_colsum_fin<<<(C + 255) / 256, 256, 0, s>>>(C, part, out);
        };
        const size_t counts = (size_t)(A + 1) * 4;
        if (counts > 48 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(k_bw_rowsort, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)counts);
            if (e != cudaSuccess) return e;
        }
        k_bw_rowsort<<<CHUNKS, 256, counts, s>>>(NT, A, actions, srows, soff);
        k_bw_arows<<<dim3(A + 1, CHUNKS), 256, 0, s>>>(NT, A, H4, srows, soff, dG, apart);
        k_bw_arows_fin<<<grid_of((size_t)A * H4), 256, 0, s>>>(A, H4, apart, g.W_lstm + (size_t)Z * H4);
        colsum((size_t)CHUNKS * (A + 1), H4, apart, g.b_lstm);
        colsum(NT, M, dMD, g.b_mdn);
        launches += 7;
    }
    h->last_launches += launches;
    return cudaGetLastError();
}

cudaError_t wm_bw_launch(const wm_handle *h, int N, int T, const float *z_seq, const int32_t *actions,
                         const int32_t *lengths, const wm_grads &g, const wm_bw_fwd &f, void *tail, cudaStream_t s) {
    if (N == 0 || T == 0) {  // no rows: every gradient is 0
        const wm_config &c = h->cfg;
        const size_t Z = c.z_dim, A = c.a_dim, H = c.h_dim, M = h->M;
        cudaError_t e = cudaMemsetAsync(g.W_lstm, 0, (Z + A + H) * 4 * H * 4, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(g.b_lstm, 0, 4 * H * 4, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(g.W_mdn, 0, H * M * 4, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(g.b_mdn, 0, M * 4, s);
        return e;
    }
    if (h->cfg.precision == WM_BF16)
        return bw_run<__nv_bfloat16>(h, N, T, z_seq, actions, lengths, g, f, (char *)tail, s);
    return bw_run<float>(h, N, T, z_seq, actions, lengths, g, f, (char *)tail, s);
}
