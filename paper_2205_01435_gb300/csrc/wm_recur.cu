// wm_recur.cu -- the teacher-forced LSTM recurrence as one persistent kernel: all T steps of
// X_t = [z_t | h_t] x W_g + W_a[a_t] + b -> cell -> h_{t+1} in one launch (Sec. 3.3.2).
//
// The recurrence is a chain of T small products, bound by what lies between them and not by
// the tensor pipe.  As one launch per step (512 sequences, H = 512) a step took 9.0 us: the
// launch hand-off 2.1, the wait for the first operands 1.3, two rounds of operand loads 3.1
// and the epilogue 2.5.  Here every CTA keeps its share of the gate weights in shared memory
// for all T steps, and the hand-off is a counter:
//   - a CTA owns a unit tile (U hidden units, all four gates: 4U columns, resident) and a row
//     tile of 128 sequences (M = 128 tcgen05 MMAs), or several row tiles in turn when there are
//     more than the SMs hold; the cell state c stays in its shared memory;
//   - h_{t+1} goes to the operand rows of frame t + 1 in global memory (L2), then the CTA adds
//     one to the row tile's counter (release); the CTAs of that row tile load their rows by TMA
//     once the counter shows all unit tiles of step t (acquire).  Frames are distinct rows, so
//     nothing is overwritten and one counter is the only dependency.  Every CTA loads its whole
//     operand blocks itself.
// A step (512 sequences, H = 512) takes about 4 us: operands through L2, MMAs, cell, stores and the
// hand-off are one chain.  A call of 512 x 128 takes 0.65 ms, 1.28 as one launch per step; on the
// fp32 path (two parts per block through a ring that holds 4; paced by the issuer's MMAs) 1.22 ms,
// 2.38 before.  (With the loads of a row tile shared by a cluster of four CTAs: 0.67 and 1.21.)  Up
// to RECUR_MAX_GROUPS row tiles per CTA this stays ahead of one launch per step (24 steps at H = 512:
// 1024 / 2048 sequences 221 / 341 us against 288 / 432).
// Every CTA waits for others: the launch is cooperative (all CTAs resident), every wait is
// bounded, and a CTA that gives up records WM_ERR_TIMEOUT and exits: its epilogue leaves the step loop
// at the barrier before the counter's release, all warps together, so that the CTAs that wait for the
// counter give up in their turn.
//
// Warps: 0 the TMA producer, 1 the MMA issuer (and TMEM), 2..9 the epilogue (two warps per TMEM
// lane quadrant, U / 2 units each).  TMEM holds two accumulators of 4U columns (fp32 path: 8U).
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>

#include "tc_ptx.cuh"
#include "wm_device.cuh"
#include "wm_internal.h"

using namespace wmk;

namespace {

constexpr int BM = 128, BK = 64;
constexpr int EPI_THREADS = 256, THREADS = 64 + EPI_THREADS;
constexpr uint32_t A_BYTES = BM * BK * 2;
constexpr uint32_t POLLS = 1u << 24, FLAG_POLLS = 1u << 21;  // mbarrier polls; counter polls (about 1 s)
constexpr int MAX_STAGES = 16;

__device__ __forceinline__ int ld_acquire(const int *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// generic-proxy global accesses ordered before / after TMA's (async-proxy) ones
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

__device__ __forceinline__ float tanh_hw(float x) {
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// MODE 0: bf16 operands, hardware tanh; 1: bf16 operands, the stepwise family's accurate
// nonlinearities; 2: the fp32 path, each operand as bf16 hi and lo parts (products hi.hi + hi.lo +
// lo.hi), accurate tanh.
// KPS operand parts (16 KB) make a ring stage: the producer's and the issuer's turns cost 200 to 300
// cycles a stage beside the copies (30 each) and MMAs (70 a part), and a part lands every 215.
template <int MODE, int U, int KPS>
__global__ void __launch_bounds__(THREADS, 1)
    k_recur(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmXl,
            const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmWl, wm_recur_args p) {
    constexpr bool F32 = MODE == 2;
    constexpr int PARTS = F32 ? 2 : 1, UT = U / 2, N = 4 * U;
    // The fp32 path's weights of a block are 2N rows in shared memory, hi above lo: A's hi part meets both
    // in one MMA of 2N columns, hi.hi and hi.lo side by side (an MMA's time here is its operands' reads,
    // 128 bytes a cycle: 64 cycles instead of twice 48), lo.hi adds to the first half, and the
    // epilogue adds the halves.
    constexpr int NA = N * PARTS;  // columns of an accumulator
    constexpr uint32_t W_BYTES = N * BK * 2;  // one k-block of the CTA's weights
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t bar_full[MAX_STAGES], bar_empty[MAX_STAGES], bar_accf[2], bar_acce[2], bar_w, bar_done, bar_never;
    __shared__ uint32_t tmem_base;
    __shared__ int s_abort;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int n = blockIdx.x % p.n_tiles, mg = blockIdx.x / p.n_tiles;
    const int ks = p.k_steps, S = p.stages;
    const uint32_t sw = tc::smem_u32(smem), sa = sw + (uint32_t)ks * PARTS * W_BYTES;
    float *cst = reinterpret_cast<float *>(smem + (size_t)ks * PARTS * W_BYTES + (size_t)S * KPS * A_BYTES);
    auto bar = [](uint64_t *b) { return tc::smem_u32(b); };

    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            tc::mbar_init(bar(&bar_full[s]), 1);
            tc::mbar_init(bar(&bar_empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            tc::mbar_init(bar(&bar_accf[a]), 1);
            tc::mbar_init(bar(&bar_acce[a]), EPI_THREADS / 32);
        }
        tc::mbar_init(bar(&bar_w), 1);
        tc::mbar_init(bar(&bar_done), 1);
        tc::mbar_init(bar(&bar_never), 1);
        tc::fence_mbar_init();
        s_abort = 0;
    }
    if (warp == 1) tc::tmem_alloc(tc::smem_u32(&tmem_base), 2 * NA);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tm = tmem_base;
    int T = p.T;
    // injected wait (tests of the timeout path): every CTA gives up before it issues anything
    if (p.test_wait) {
        if (tid == 0 && !tc::mbar_wait_bounded(bar(&bar_never), 0, p.test_wait)) {
            s_abort = 1;
            atomicExch(p.status, (int)WM_ERR_TIMEOUT);
        }
        __syncthreads();
        if (s_abort) T = 0;
    }
    // Waits of a whole warp: one try in line (the usual case), then polls that also watch for another
    // warp's giving up.  False once anybody gave up.
    auto wait_slow = [&](uint64_t *b, uint32_t parity) {
        for (uint32_t i = 0; i < POLLS; ++i) {
            if (tc::mbar_try_wait(bar(b), parity)) return true;
            if (*(volatile int *)&s_abort) return false;
        }
        s_abort = 1;
        atomicExch(p.status, (int)WM_ERR_TIMEOUT);
        return false;
    };
    auto wait = [&](uint64_t *b, uint32_t parity) {
        bool ok = tc::mbar_try_wait(bar(b), parity);
        if (!ok) ok = wait_slow(b, parity);
        return __all_sync(0xffffffffu, ok);
    };
    const int np = ks * PARTS;  // operand parts per tile: block kb's hi (and, fp32 path, lo) part
    if (warp == 0) {
        if (T > 0) {  // ---- TMA producer (the whole warp runs the loop, one lane issues)
            if (tc::elect_one()) tc::mbar_arrive_expect_tx(bar(&bar_w), (uint32_t)np * W_BYTES);
            for (int i = 0; i < np; ++i)
                for (int gate = 0; gate < 4; ++gate)  // the 128-column packing: rows 128 j + 32 gate + u
                    if (tc::elect_one())
                        tc::tma_load_2d(sw + i * W_BYTES + gate * U * BK * 2, i % PARTS ? &tmWl : &tmW, i / PARTS * BK,
                                        U == 32 ? 128 * n + 32 * gate : 128 * (n >> 1) + 32 * gate + 16 * (n & 1), bar(&bar_w));
            int stage = 0, used = 0;
            uint32_t phase = 0;
            bool go = true;
            for (int t = 0; t < T && go; ++t)
                for (int m = mg; m < p.m_tiles && go; m += p.m_groups) {
                    if (t > 0) {  // h_t: every unit tile of step t - 1
                        bool ok = false;
                        for (uint32_t i = 0; i < FLAG_POLLS && !ok && !s_abort; ++i) ok = ld_acquire(p.count + m) >= p.n_tiles * t;
                        if (!ok && !s_abort) {
                            s_abort = 1;
                            atomicExch(p.status, (int)WM_ERR_TIMEOUT);
                        }
                        if (!__all_sync(0xffffffffu, ok)) break;
                        fence_proxy_async_global();
                    }
                    const int y = t * p.N + m * BM;
                    for (int i0 = 0; i0 < np; i0 += KPS) {
                        const int nk = np - i0 < KPS ? np - i0 : KPS;
                        if (!(go = wait(&bar_empty[stage], phase ^ 1u))) break;
                        if (tc::elect_one()) {
                            const uint32_t full = bar(&bar_full[stage]), dst = sa + stage * KPS * A_BYTES;
                            tc::mbar_arrive_expect_tx(full, nk * A_BYTES);
#pragma unroll
                            for (int h = 0; h < KPS; ++h)
                                if (h < nk)
                                    tc::tma_load_2d(dst + h * A_BYTES, F32 && (h & 1) ? &tmXl : &tmX, (i0 + h) / PARTS * BK, y, full);
                        }
                        ++used;
                        if (++stage == S) { stage = 0; phase ^= 1u; }
                    }
                }
            // nothing may be in flight into shared memory when the CTA exits
            __syncwarp();
            tc::mbar_wait_bounded(bar(&bar_w), 0, POLLS);
            for (int i = used > S ? used - S : 0; i < used; ++i)
                tc::mbar_wait_bounded(bar(&bar_full[i % S]), (uint32_t)(i / S) & 1u, POLLS);
        }
    } else if (warp == 1) {
        if (T > 0) {  // ---- MMA issuer (likewise)
            bool go = wait(&bar_w, 0);
            int stage = 0, acc = 0;
            uint32_t phase = 0, acc_phase = 0;
            const uint32_t idesc = tc::idesc_bf16_f32(BM, N), idesc2 = tc::idesc_bf16_f32(BM, NA);
            for (int t = 0; t < T && go; ++t)
                for (int m = mg; m < p.m_tiles && go; m += p.m_groups) {
                    if (!(go = wait(&bar_acce[acc], acc_phase ^ 1u))) break;
                    tc::fence_after_sync();
                    const uint32_t d = tm + acc * NA;
                    for (int i0 = 0; i0 < np; i0 += KPS) {
                        const int nk = np - i0 < KPS ? np - i0 : KPS;
                        if (!(go = wait(&bar_full[stage], phase))) break;
                        tc::fence_after_sync();
                        if (tc::elect_one()) {
                            const uint64_t da0 = tc::desc_sw128(sa + stage * KPS * A_BYTES), db0 = tc::desc_sw128(sw + i0 * W_BYTES);
#pragma unroll
                            for (int h = 0; h < KPS; h += PARTS) {
                                if (h >= nk) break;
                                const uint64_t da = da0 + h * (A_BYTES >> 4), db = db0 + h * (W_BYTES >> 4);
#pragma unroll
                                for (int kk = 0; kk < BK / 16; ++kk)
                                    tc::mma_bf16(d, da + 2 * kk, db + 2 * kk, idesc2, (i0 + h > 0 || kk > 0) ? 1u : 0u);
                                if (F32) {
#pragma unroll
                                    for (int kk = 0; kk < BK / 16; ++kk)  // lo . hi
                                        tc::mma_bf16(d, da + (A_BYTES >> 4) + 2 * kk, db + 2 * kk, idesc, 1u);
                                }
                            }
                            tc::mma_commit(bar(&bar_empty[stage]));
                        }
                        if (++stage == S) { stage = 0; phase ^= 1u; }
                    }
                    if (tc::elect_one()) tc::mma_commit(bar(&bar_accf[acc]));
                    acc ^= 1;
                    if (acc == 0) acc_phase ^= 1u;
                }
            __syncwarp();
            if (tc::elect_one()) tc::mma_commit(bar(&bar_done));  // no MMA in flight when TMEM is freed
            tc::mbar_wait_bounded(bar(&bar_done), 0, POLLS);
        }
    } else {  // ---- epilogue
        const int quad = warp & 3, half = (warp - 2) >> 2, r = 32 * quad + lane;
        const int u0 = UT * half, ug = U * n + u0;  // the thread's first unit: in the tile, in H
        // the tile's columns in the 128-column packing (bias, action rows)
        const int col0 = U == 32 ? 128 * n : 128 * (n >> 1) + 16 * (n & 1);
        float bias[4][UT];
#pragma unroll
        for (int g = 0; g < 4; ++g)
#pragma unroll
            for (int j = 0; j < UT; ++j) bias[g][j] = p.bias[col0 + 32 * g + u0 + j];
        for (int gi = 0, m = mg; m < p.m_tiles; ++gi, m += p.m_groups)
#pragma unroll
            for (int j = 0; j < UT; ++j) cst[((size_t)gi * U + u0 + j) * BM + r] = 0.f;
        int acc = 0;
        uint32_t acc_phase = 0;
        // UT units of an output row: whole 32-byte sectors where the row's start and length allow
        const bool whole = (p.H & 7) == 0 && ((reinterpret_cast<uintptr_t>(p.h_seq) | reinterpret_cast<uintptr_t>(p.c_seq)) & 31) == 0;
        auto store_row = [&](float *q, const float (&v)[UT], int nu) {
#pragma unroll
            for (int j0 = 0; j0 < UT; j0 += 8) {
                if (whole) {
                    if (j0 < nu)  // (nu is a multiple of 8, or not positive)
                        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                                     :: "l"(q + j0), "f"(v[j0]), "f"(v[j0 + 1]), "f"(v[j0 + 2]), "f"(v[j0 + 3]), "f"(v[j0 + 4]),
                                        "f"(v[j0 + 5]), "f"(v[j0 + 6]), "f"(v[j0 + 7]) : "memory");
                } else {
#pragma unroll
                    for (int j = j0; j < j0 + 8; ++j)
                        if (j < nu) q[j] = v[j];
                }
            }
        };
        auto sig = [](float x) {
            return MODE == 1 ? sigmoid_newton(x) : MODE ? fmaf(0.5f, tanhf(0.5f * x), 0.5f) : fmaf(0.5f, tanh_hw(0.5f * x), 0.5f);
        };
        auto th = [](float x) { return MODE ? tanhf(x) : tanh_hw(x); };
        // The action row's columns are gathers from L2 (32 lines per load).  They go out right after a
        // tile's h' (its action was loaded one tile before that), so that they are done before the next
        // tile's operands arrive: under those they hold up the producer's and the issuer's own accesses.
        uint32_t w[PARTS][4][UT / 2];
        auto act_of = [&](int t, int m) {
            const int b = m * BM + r;
            return t < T ? p.act[(size_t)t * p.N + (b < p.N ? b : 0)] : -1;
        };
        auto gather = [&](int t, int m, int a) {
            if (t >= T) return;
            if (a >= p.A && m * BM + r < p.N && n == 0 && half == 0) report_status(p.status, WM_ERR_INVALID_ARG);
            const bool some = a >= 0 && a < p.A;
#pragma unroll
            for (int q = 0; q < PARTS; ++q)
#pragma unroll
                for (int g = 0; g < 4; ++g)
#pragma unroll
                    for (int j = 0; j < UT / 8; ++j) {
                        uint4 v = make_uint4(0u, 0u, 0u, 0u);
                        if (some)
                            v = __ldg(reinterpret_cast<const uint4 *>((q ? p.wa_lo : p.wa) + (size_t)a * 4 * p.Hp + col0 + 32 * g +
                                                                      u0 + 8 * j));
                        w[q][g][4 * j] = v.x; w[q][g][4 * j + 1] = v.y; w[q][g][4 * j + 2] = v.z; w[q][g][4 * j + 3] = v.w;
                    }
        };
        int t1 = 0, m1 = mg;  // the tile after the one whose action is in a1
        auto advance = [&] {
            m1 += p.m_groups;
            if (m1 >= p.m_tiles) { m1 = mg; ++t1; }
        };
        int a1 = act_of(t1, m1);
        gather(t1, m1, a1);
        advance();
        a1 = act_of(t1, m1);
        bool go = true;
        for (int t = 0; t < T && go; ++t)
            for (int gi = 0, m = mg; m < p.m_tiles; ++gi, m += p.m_groups) {
                const int b = m * BM + r;
                const bool valid = b < p.N;
                const size_t row = (size_t)t * p.N + (valid ? b : 0);
                const bool ok = wait(&bar_accf[acc], acc_phase);
                __syncwarp();
                tc::fence_after_sync();
                const uint32_t ta = tm + ((uint32_t)(32 * quad) << 16) + acc * NA + u0;
                float c[UT], h[UT];
                const size_t o = row * p.H + ug;
                const int nu = p.H - ug;  // units from ug on that are not padding
                float pre[4][8];  // eight units' gate pre-activations (for g_seq)
                // (asked for with H % 8 == 0 and aligned rows only)
                auto store_pre = [&](int j0) {
                    if (!valid || !p.g_seq || j0 >= nu) return;
                    float *q = p.g_seq + 4 * row * p.H + ug + j0;
#pragma unroll
                    for (int g = 0; g < 4; ++g, q += p.H)
                        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                                     :: "l"(q), "f"(pre[g][0]), "f"(pre[g][1]), "f"(pre[g][2]), "f"(pre[g][3]), "f"(pre[g][4]),
                                        "f"(pre[g][5]), "f"(pre[g][6]), "f"(pre[g][7]) : "memory");
                };
#pragma unroll
                for (int j0 = 0; j0 < UT; j0 += 8) {
                    uint32_t v[4][8];
#pragma unroll
                    for (int g = 0; g < 4; ++g) TC_LD8(ta + U * g + j0, v[g]);
                    tc::tmem_ld_wait();
                    if (F32) {
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            uint32_t v2[8];
                            TC_LD8(ta + N + U * g + j0, v2);
                            tc::tmem_ld_wait();
#pragma unroll
                            for (int j = 0; j < 8; ++j) v[g][j] = __float_as_uint(__uint_as_float(v[g][j]) + __uint_as_float(v2[j]));
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float x[4];
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            const uint32_t wv = w[0][g][(j0 + j) / 2];
                            x[g] = __uint_as_float(v[g][j]) + bias[g][j0 + j] + __uint_as_float((j & 1) ? wv & 0xffff0000u : wv << 16);
                            if (F32) {
                                const uint32_t wl = w[PARTS - 1][g][(j0 + j) / 2];
                                x[g] += __uint_as_float((j & 1) ? wl & 0xffff0000u : wl << 16);
                            }
                            pre[g][j] = x[g];
                        }
                        float &cs = cst[((size_t)gi * U + u0 + j0 + j) * BM + r];
                        const float cv = sig(x[1]) * cs + sig(x[0]) * th(x[2]);
                        cs = cv;
                        c[j0 + j] = cv;
                        h[j0 + j] = sig(x[3]) * th(cv);
                    }
                    if (UT > 8) store_pre(j0);  // (held past the counter they would spill)
                }
                if (MODE == 1 && nu < UT) {  // a padded unit's h' is 0 also where its gates met 0 x infinity
#pragma unroll
                    for (int j = 0; j < UT; ++j) h[j] = j < nu ? h[j] : 0.f;
                }
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0)  // the accumulator may be overwritten
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(bar(&bar_acce[acc])) : "memory");
                if (valid) {  // h' into the operand rows of frame t + 1
                    const size_t xo = (row + p.N) * p.KX + p.Zp + ug;
#pragma unroll
                    for (int j0 = 0; j0 < UT; j0 += 8) {
                        uint32_t hi[4], lo[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float f0 = h[j0 + 2 * j], f1 = h[j0 + 2 * j + 1];
                            __nv_bfloat162 b2 = __floats2bfloat162_rn(f0, f1);
                            hi[j] = *reinterpret_cast<uint32_t *>(&b2);
                            if (F32) {
                                __nv_bfloat162 l2 = __floats2bfloat162_rn(f0 - __low2float(b2), f1 - __high2float(b2));
                                lo[j] = *reinterpret_cast<uint32_t *>(&l2);
                            }
                        }
                        *reinterpret_cast<uint4 *>(p.x + xo + j0) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                        if (F32) *reinterpret_cast<uint4 *>(p.x_lo + xo + j0) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                    }
                }
                fence_proxy_async_global();
                if (!(go = !tc::barrier_or(1, EPI_THREADS, !ok))) break;
                if (tid == 64)  // (the release covers the other threads' stores through the barrier)
                    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" :: "l"(p.count + m) : "memory");
                gather(t1, m1, a1);
                advance();
                a1 = act_of(t1, m1);
                // the optional outputs, off the chain
                if (UT == 8) store_pre(0);
                if (valid && p.h_seq) store_row(p.h_seq + o, h, nu);
                if (valid && p.c_seq) store_row(p.c_seq + o, c, nu);
                acc ^= 1;
                if (acc == 0) acc_phase ^= 1u;
            }
    }
    __syncwarp();
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) tc::tmem_dealloc(tm, 2 * NA);
}

constexpr size_t SMEM_MAX = 227 * 1024, SMEM_STATIC = 1024;

// shared memory beside the ring, per CTA
size_t fixed_smem(bool f32, int U, int ks, int groups) {
    return 1024 + (size_t)ks * (f32 ? 2 : 1) * 4 * U * BK * 2 + (size_t)groups * U * BM * 4;
}

using kern_t = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, wm_recur_args);
kern_t kernel_of(int mode, int units, int kps) {
    if (mode == 2) return units == 16 ? k_recur<2, 16, 2> : k_recur<2, 32, 2>;
    if (mode == 1)
        return units == 16 ? (kps == 3 ? k_recur<1, 16, 3> : k_recur<1, 16, 2>) : (kps == 3 ? k_recur<1, 32, 3> : k_recur<1, 32, 2>);
    return units == 16 ? (kps == 3 ? k_recur<0, 16, 3> : k_recur<0, 16, 2>) : (kps == 3 ? k_recur<0, 32, 3> : k_recur<0, 32, 2>);
}

}  // namespace

// The CTAs that can be resident at once (one per SM), and the kernels' shared-memory limit on this device.
cudaError_t wm_recur_prepare(wm_handle *h) {
    if (h->recur_ready || !h->tc.ok) return cudaSuccess;
    const bool f32 = h->cfg.precision == WM_FP32;
    const size_t smem = SMEM_MAX - SMEM_STATIC;
    cudaError_t e = cudaSuccess;
    for (int mode = f32 ? 2 : 0; mode < (f32 ? 3 : 2); ++mode)
        for (int units : {16, 32})
            for (int kps = 2; kps <= (f32 ? 2 : 3); ++kps) {
                const kern_t kern = kernel_of(mode, units, kps);
                int n = 0;
                if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, THREADS, smem);
                h->recur_ctas[mode][units >> 5][kps - 2] = n * h->sms;
            }
    h->recur_ready = e == cudaSuccess;
    return e;
}

bool wm_recur_plan(const wm_handle *h, int mode, int N, int Hp, int KX, wm_recur_args *a) {
    const bool f32 = mode == 2;
    const int ks = (KX + BK - 1) / BK, mt = (N + BM - 1) / BM;
    bool found = false;
    for (int U : {16, 32}) {
        const int nt = Hp / U;
        // the ring's depth follows from what the weights and the cell states leave
        int mg = 0, groups = 0, kps = 0, stages = 0;
        size_t fixed = 0;
        for (int pass = 0; pass < 2; ++pass) {  // (the states' share depends on the resident CTAs, found with kps = 2)
            const int ctas = h->recur_ctas[mode][U >> 5][pass ? kps - 2 : 0];
            if (nt > ctas) { stages = 0; break; }
            mg = mt < ctas / nt ? mt : ctas / nt;
            groups = (mt + mg - 1) / mg;
            fixed = fixed_smem(f32, U, ks, groups) + SMEM_STATIC;
            const int parts = fixed < SMEM_MAX ? (int)((SMEM_MAX - fixed) / A_BYTES) : 0;
            kps = !f32 && parts >= 9 ? 3 : 2;
            stages = parts / kps < MAX_STAGES ? parts / kps : MAX_STAGES;
        }
        if (stages < 2 || groups > RECUR_MAX_GROUPS || (found && groups >= a->groups)) continue;
        found = true;
        a->units = U;
        a->n_tiles = nt;
        a->m_tiles = mt;
        a->m_groups = mg;
        a->groups = groups;
        a->k_steps = ks;
        a->stages = stages;
        a->kps = kps;
        a->smem = fixed - SMEM_STATIC + (size_t)stages * kps * A_BYTES;
    }
    return found;
}

cudaError_t wm_recur_launch(int mode, const void *x_map, const void *xl_map, const void *w_map, const void *wl_map,
                            const wm_recur_args &a, cudaStream_t s) {
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;  // every CTA resident: they wait for one another
    at[0].val.cooperative = 1;
    lc.gridDim = dim3((unsigned)(a.n_tiles * a.m_groups));
    lc.blockDim = dim3(THREADS);
    lc.dynamicSmemBytes = a.smem;
    lc.stream = s;
    lc.attrs = at;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, kernel_of(mode, a.units, a.kps), *(const CUtensorMap *)x_map, *(const CUtensorMap *)xl_map,
                              *(const CUtensorMap *)w_map, *(const CUtensorMap *)wl_map, a);
}
