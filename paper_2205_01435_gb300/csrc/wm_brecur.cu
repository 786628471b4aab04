// wm_brecur.cu -- the training step's backward recurrence as one persistent kernel: for t = T-1 .. 0
//   dH_t = dG_{t+1} W_h^T,  dh = dY_t + dH_t,  the cell's backward step -> dG_t      (Sec. 3.3.2)
// in one launch (as two launches per step, a cell kernel and a library GEMM, a step took 11.8 us at
// 512 sequences and H = 512, almost all of it latency; about 7 us here; clock64 stamps of one CTA: counter to product
// 3.9K cycles, exchange 2.9K, cell 0.9K, stores and the counter's release 3.3K, release to acquire 1.7K).
//
// The product contracts over 4H gate columns, four times what the forward's does, so a CTA could not
// stream its rows' operands in time (512 KB a step at about 77 B per cycle).  A cluster of four CTAs
// therefore splits the contraction by gate: CTA g of a cluster
//   - keeps the gate's part of W_h for 64 units in shared memory (64 rows x H, K-major),
//   - loads gate g's columns of dG_{t+1} for its 128 rows by TMA and forms a 128 x 64 partial product
//     (tcgen05, fp32 in TMEM),
//   - sends the partials of the other CTAs' 16 units into their shared memory (st.async, counted on
//     the receiver's mbarrier), and sums the four partials of its own 16 units in gate order
//     (deterministic),
//   - does the cell's backward step for its 128 rows x 16 units, with the carried dc and c in
//     registers, stores dG_t and adds one to the row tile's counter, which the loads of step t - 1
//     wait for (as in wm_recur.cu).
// The activations (or pre-activations), c and dY of the step are loaded before the wait for the
// product, and prefetched into L2 a step earlier (without: 3338 instead of 3221 us per training step).  Every CTA
// waits for others: cooperative launch, bounded waits, WM_ERR_TIMEOUT on giving up.  A CTA that gives up
// sends no partials that it has not computed, arms no barrier again and releases no counter: its epilogue
// leaves the step loop at one of the two barriers of a step, all warps together, and the CTAs that wait
// for it give up in their turn.  Before its cluster's last barrier it gives the partials under way, its
// own and its peers', time to land.
//
// F32: the operands are bf16 hi and lo parts (dG_t's in a two-step ring of their own, W_h's packed
// once) and the products hi.hi + hi.lo + lo.hi, as everywhere on the fp32 path.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>

#include "tc_ptx.cuh"
#include "wm_internal.h"

namespace {

constexpr int BM = 128, BK = 64, CL = 4, UC = 64, U = UC / CL;  // rows; k-block; CTAs, units per cluster; units per CTA
constexpr int EPI_THREADS = 256, THREADS = 64 + EPI_THREADS;
constexpr uint32_t A_BYTES = BM * BK * 2, W_BYTES = UC * BK * 2, SLOT = BM * U * 4;  // one gate's partials: 8 KB
constexpr uint32_t POLLS = 1u << 24, FLAG_POLLS = 1u << 21;
constexpr int MAX_STAGES = 8, KPS = 2;  // ring stages of two operand parts (see wm_recur.cu)

__device__ __forceinline__ int ld_acquire(const int *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ void st_async16(uint32_t dst, float4 v, uint32_t mbar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 :: "r"(dst), "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)),
                    "r"(__float_as_uint(v.w)), "r"(mbar) : "memory");
}
// eight floats at a 32-byte boundary: one sector per lane
__device__ __forceinline__ void ld32(const float *p, float (&v)[8]) {
    asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "l"(p));
}
__device__ __forceinline__ void st32(float *p, const float (&v)[8]) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 :: "l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
}
// byte offset of 16-byte chunk c (0..3) of row r in a slot: rows of 64 bytes, chunks permuted so that
// eight consecutive rows' accesses to one chunk fall on distinct banks
__device__ __forceinline__ uint32_t slot_at(int r, int c) { return r * 64 + ((c ^ ((r >> 1) & 3)) << 4); }

template <bool F32>
__global__ void __launch_bounds__(THREADS, 1)
    k_brecur(const __grid_constant__ CUtensorMap tmG, const __grid_constant__ CUtensorMap tmW, wm_brecur_args p) {
    constexpr int PARTS = F32 ? 2 : 1;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t bar_full[MAX_STAGES], bar_empty[MAX_STAGES], bar_acc, bar_x, bar_w, bar_done, bar_never;
    __shared__ uint32_t tmem_base;
    __shared__ int s_abort;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int g = (int)tc::cluster_rank(), cl = blockIdx.x / CL, uj = cl % p.u_tiles, m = p.m0 + cl / p.u_tiles;
    const int H = p.H, H4 = 4 * H, ks = H / BK, np = ks * PARTS, S = p.stages, N = p.N;
    const uint32_t sw = tc::smem_u32(smem), sa = sw + (uint32_t)np * W_BYTES, sx = sa + (uint32_t)S * KPS * A_BYTES;
    const unsigned char *xbuf = smem + (size_t)np * W_BYTES + (size_t)S * KPS * A_BYTES;
    auto bar = [](uint64_t *b) { return tc::smem_u32(b); };
    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            tc::mbar_init(bar(&bar_full[s]), 1);
            tc::mbar_init(bar(&bar_empty[s]), 1);
        }
        for (uint64_t *b : {&bar_acc, &bar_x, &bar_w, &bar_done, &bar_never}) tc::mbar_init(bar(b), 1);
        tc::fence_mbar_init();
        s_abort = 0;
    }
    if (warp == 1) tc::tmem_alloc(tc::smem_u32(&tmem_base), UC * PARTS);
    tc::fence_before_sync();
    tc::cluster_sync();  // the cluster's barriers exist before any store reaches them
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
    auto wait_slow = [&](uint64_t *b, uint32_t parity) {
        for (uint32_t i = 0; i < POLLS; ++i) {
            if (tc::mbar_try_wait(bar(b), parity)) return true;
            if (*(volatile int *)&s_abort) return false;
        }
        s_abort = 1;
        atomicExch(p.status, (int)WM_ERR_TIMEOUT);
        return false;
    };
    auto wait = [&](uint64_t *b, uint32_t parity) {  // a whole warp; false once anybody gave up
        bool ok = tc::mbar_try_wait(bar(b), parity);
        if (!ok) ok = wait_slow(b, parity);
        return __all_sync(0xffffffffu, ok);
    };

    if (T == 0) {
        // (gave up, or nothing to do)
    } else if (warp == 0) {  // ---- TMA producer
        if (tc::elect_one()) tc::mbar_arrive_expect_tx(bar(&bar_w), (uint32_t)np * W_BYTES);
        for (int i = 0; i < np; ++i)  // W_h: rows of units, gate g's columns (lo parts 4H further)
            if (tc::elect_one())
                tc::tma_load_2d(sw + i * W_BYTES, &tmW, (i % PARTS) * H4 + g * H + i / PARTS * BK, p.w_row0 + UC * uj, bar(&bar_w));
        int stage = 0, used = 0;
        uint32_t phase = 0;
        bool go = true;
        for (int t = T - 2; t >= 0 && go; --t) {
            const int want = p.u_tiles * CL * (T - 1 - t);  // every unit of dG_{t+1}
            bool ok = false;
            for (uint32_t i = 0; i < FLAG_POLLS && !ok && !s_abort; ++i) ok = ld_acquire(p.count + m) >= want;
            if (!ok && !s_abort) {
                s_abort = 1;
                atomicExch(p.status, (int)WM_ERR_TIMEOUT);
            }
            if (!(go = __all_sync(0xffffffffu, ok))) break;
            fence_proxy_async_global();
            const int y = (F32 ? ((t + 1) & 1) * N : (t + 1) * N) + m * BM;
            for (int i0 = 0; i0 < np; i0 += KPS) {
                const int nk = np - i0 < KPS ? np - i0 : KPS;
                if (!(go = wait(&bar_empty[stage], phase ^ 1u))) break;
                if (tc::elect_one()) {
                    const uint32_t full = bar(&bar_full[stage]), dst = sa + stage * KPS * A_BYTES;
                    tc::mbar_arrive_expect_tx(full, nk * A_BYTES);
#pragma unroll
                    for (int h = 0; h < KPS; ++h)
                        if (h < nk)
                            tc::tma_load_2d(dst + h * A_BYTES, &tmG, (F32 && h ? H4 : 0) + g * H + (i0 + h) / PARTS * BK, y, full);
                }
                ++used;
                if (++stage == S) { stage = 0; phase ^= 1u; }
            }
        }
        // no copy of this CTA's may be in flight into its shared memory when it exits
        __syncwarp();
        tc::mbar_wait_bounded(bar(&bar_w), 0, POLLS);
        for (int i = used > S ? used - S : 0; i < used; ++i)
            tc::mbar_wait_bounded(bar(&bar_full[i % S]), (uint32_t)(i / S) & 1u, POLLS);
    } else if (warp == 1) {  // ---- MMA issuer
        bool go = wait(&bar_w, 0);
        int stage = 0;
        uint32_t phase = 0;
        // (fp32 path: hi meets hi and lo in one MMA, see wm_recur.cu)
        const uint32_t idesc = tc::idesc_bf16_f32(BM, UC), idesc2 = tc::idesc_bf16_f32(BM, UC * PARTS);
        for (int t = T - 2; t >= 0 && go; --t) {
            // (the accumulator is free: dG_{t+1}'s counter covers this CTA's reads of it)
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
                            tc::mma_bf16(tm, da + 2 * kk, db + 2 * kk, idesc2, (i0 + h > 0 || kk > 0) ? 1u : 0u);
                        if (F32) {
#pragma unroll
                            for (int kk = 0; kk < BK / 16; ++kk)  // lo . hi
                                tc::mma_bf16(tm, da + (A_BYTES >> 4) + 2 * kk, db + 2 * kk, idesc, 1u);
                        }
                    }
                    tc::mma_commit(bar(&bar_empty[stage]));
                }
                if (++stage == S) { stage = 0; phase ^= 1u; }
            }
            if (tc::elect_one()) tc::mma_commit(bar(&bar_acc));
        }
        __syncwarp();
        if (tc::elect_one()) tc::mma_commit(bar(&bar_done));  // no MMA in flight when TMEM is freed
        tc::mbar_wait_bounded(bar(&bar_done), 0, POLLS);
    } else {  // ---- epilogue
        // Of the product a thread reads 32 columns of accumulator row r (TMEM fixes the row by lane).
        // Of the cell it takes row e / 2 and 8 units, so that two lanes cover a row's 16 units: every
        // global access is whole 32-byte sectors (with a row per lane they were halves, and the stores
        // took 3K cycles to complete before the counter's release).
        const int quad = warp & 3, half = (warp - 2) >> 2, r = 32 * quad + lane;
        const int e = tid - 64, er = e >> 1, eh = e & 1;
        const int u = UC * uj + U * g + 8 * eh;  // the thread's first unit
        const bool valid = m * BM + er < N;
        const int n = valid ? m * BM + er : 0;
        float dc[8], c[8];  // dc carried from step t + 1; c_t
#pragma unroll
        for (int j = 0; j < 8; ++j) dc[j] = 0.f;
        struct In {
            float ig[8], fg[8], gg[8], og[8], cp[8], dh[8];
        };
        In in;
        auto load = [&](int t, In &v) {  // step t's activations, dY and c_{t-1}
            const size_t row = (size_t)t * N + n;
            const float *a = p.act + row * H4 + u;
            ld32(a, v.ig);
            ld32(a + H, v.fg);
            ld32(a + 2 * H, v.gg);
            ld32(a + 3 * H, v.og);
            ld32(p.dY + row * H + u, v.dh);
            if (t > 0) {
                ld32(p.cs + (row - N) * H + u, v.cp);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) v.cp[j] = 0.f;
            }
        };
        auto fetch = [&](int t) {  // the same of a later step into L2: the loads then don't wait for DRAM
            const size_t row = (size_t)t * N + n;
            const float *a = p.act + row * H4 + u;
#pragma unroll
            for (int q = 0; q < 4; ++q) asm volatile("prefetch.global.L2 [%0];" :: "l"(a + q * H));
            asm volatile("prefetch.global.L2 [%0];" :: "l"(p.dY + row * H + u));
            if (t > 0) asm volatile("prefetch.global.L2 [%0];" :: "l"(p.cs + (row - N) * H + u));
        };
        ld32(p.cs + ((size_t)(T - 1) * N + n) * H + u, c);
        load(T - 1, in);
        uint32_t ph = 0;
        bool ok = true;
        for (int t = T - 1; t >= 0; --t) {
            const size_t row = (size_t)t * N + n;
            if (p.pre) {  // the activations, under the wait for the product
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    in.ig[j] = 1.f / (1.f + expf(-in.ig[j]));
                    in.fg[j] = 1.f / (1.f + expf(-in.fg[j]));
                    in.gg[j] = tanhf(in.gg[j]);
                    in.og[j] = 1.f / (1.f + expf(-in.og[j]));
                }
            }
            if (t < T - 1) {
                if (tid == 64) tc::mbar_arrive_expect_tx(bar(&bar_x), (CL - 1) * SLOT);
                ok = wait(&bar_acc, ph);
                tc::fence_after_sync();
                float v[32];
                {
                    uint32_t q[32];
                    const uint32_t ta = tm + ((uint32_t)(32 * quad) << 16) + 32 * half;
                    TC_LD16(ta, q);
                    TC_LD16(ta + 16, (q + 16));
                    tc::tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(q[j]);
                    if (F32) {
                        TC_LD16(ta + UC, q);
                        TC_LD16(ta + UC + 16, (q + 16));
                        tc::tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] += __uint_as_float(q[j]);
                    }
                }
                tc::fence_before_sync();
#pragma unroll
                for (int s = 0; s < 2; ++s) {  // the 16 units of CTA 2 half + s: its slot g
                    const int to = 2 * half + s;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float4 q = make_float4(v[16 * s + 4 * k], v[16 * s + 4 * k + 1], v[16 * s + 4 * k + 2], v[16 * s + 4 * k + 3]);
                        const uint32_t dst = sx + g * SLOT + slot_at(r, k);
                        if (!ok) continue;
                        if (to != g) st_async16(tc::map_rank(dst, to), q, tc::map_rank(bar(&bar_x), to));
                        else *reinterpret_cast<float4 *>(const_cast<unsigned char *>(xbuf) + g * SLOT + slot_at(r, k)) = q;
                    }
                }
                if (tc::barrier_or(1, EPI_THREADS, !ok)) break;  // this CTA's own slot
                ok = wait(&bar_x, ph);
                if (ok) ph ^= 1u;  // (else the phase that is open: the drain below waits for it)
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    float4 s = *reinterpret_cast<const float4 *>(xbuf + slot_at(er, 2 * eh + k));
#pragma unroll
                    for (int q = 1; q < CL; ++q) {  // in gate order
                        const float4 a = *reinterpret_cast<const float4 *>(xbuf + q * SLOT + slot_at(er, 2 * eh + k));
                        s.x += a.x; s.y += a.y; s.z += a.z; s.w += a.w;
                    }
                    in.dh[4 * k] += s.x; in.dh[4 * k + 1] += s.y; in.dh[4 * k + 2] += s.z; in.dh[4 * k + 3] += s.w;
                }
            }
            float d[4][8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float tc_ = tanhf(c[j]);
                const float dcj = in.dh[j] * in.og[j] * (1.f - tc_ * tc_) + dc[j];
                d[0][j] = dcj * in.gg[j] * in.ig[j] * (1.f - in.ig[j]);
                d[1][j] = dcj * in.cp[j] * in.fg[j] * (1.f - in.fg[j]);
                d[2][j] = dcj * in.ig[j] * (1.f - in.gg[j] * in.gg[j]);
                d[3][j] = in.dh[j] * tc_ * in.og[j] * (1.f - in.og[j]);
                dc[j] = dcj * in.fg[j];
                c[j] = in.cp[j];
            }
            if (valid) {  // the operand rows of step t - 1's product (bf16 path: also of the weight gradients)
                __nv_bfloat16 *o = F32 ? p.parts + ((size_t)(t & 1) * N + n) * 2 * H4 + u : p.dGo + row * H4 + u;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t hi[4], lo[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        __nv_bfloat162 b2 = __floats2bfloat162_rn(d[q][2 * k], d[q][2 * k + 1]);
                        hi[k] = *reinterpret_cast<uint32_t *>(&b2);
                        if (F32) {
                            __nv_bfloat162 l2 = __floats2bfloat162_rn(d[q][2 * k] - __low2float(b2), d[q][2 * k + 1] - __high2float(b2));
                            lo[k] = *reinterpret_cast<uint32_t *>(&l2);
                        }
                    }
                    *reinterpret_cast<uint4 *>(o + q * H) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                    if (F32) *reinterpret_cast<uint4 *>(o + H4 + q * H) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                }
            }
            if (t > 0) {
                fence_proxy_async_global();
                if (tc::barrier_or(1, EPI_THREADS, !ok)) break;
                if (tid == 64)  // (the release covers the other threads' stores through the barrier)
                    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" :: "l"(p.count + m) : "memory");
                load(t - 1, in);
                if (t > 1) fetch(t - 2);
            }
            if (valid) {  // dG_t in fp32, off the chain
                float *o = p.dG + row * H4 + u;
#pragma unroll
                for (int q = 0; q < 4; ++q) st32(o + q * H, d[q]);
            }
        }
        // gave up: the phase of the partials may stay open (a peer that gave up too sends none), and then
        // the polls are the time that those under way have to land (more than a millisecond)
        if (__any_sync(0xffffffffu, !ok || s_abort)) tc::mbar_wait_bounded(bar(&bar_x), ph, 1u << 16);
    }
    __syncwarp();
    tc::fence_before_sync();
    tc::cluster_sync();  // peers' stores into this CTA's shared memory are done
    if (warp == 1) tc::tmem_dealloc(tm, UC * PARTS);
}

constexpr size_t SMEM_MAX = 227 * 1024, SMEM_STATIC = 1024;

void set_attrs(cudaLaunchConfig_t &lc, cudaLaunchAttribute (&at)[2], size_t smem) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeCooperative;
    at[1].val.cooperative = 1;
    lc.blockDim = dim3(THREADS);
    lc.dynamicSmemBytes = smem;
    lc.attrs = at;
    lc.numAttrs = 2;
}

}  // namespace

// The clusters that can be resident at once, and the kernel's shared-memory limit on this device.
cudaError_t wm_brecur_prepare(wm_handle *h) {
    if (h->brecur_ready || h->cfg.h_dim % UC) return cudaSuccess;
    const bool f32 = h->cfg.precision == WM_FP32;
    const void *kern = f32 ? (const void *)k_brecur<true> : (const void *)k_brecur<false>;
    const size_t smem = SMEM_MAX - SMEM_STATIC;
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[2];
    set_attrs(lc, at, smem);
    lc.gridDim = dim3(CL);
    lc.numAttrs = 1;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&h->brecur_clusters, kern, &lc);
    h->brecur_ready = e == cudaSuccess;
    return e;
}

bool wm_brecur_plan(const wm_handle *h, int N, int H, wm_brecur_args *a) {
    if (H % UC) return false;
    const bool f32 = h->cfg.precision == WM_FP32;
    const int np = H / BK * (f32 ? 2 : 1), clusters = h->brecur_clusters;
    a->u_tiles = H / UC;
    a->m_tiles = (N + BM - 1) / BM;
    const size_t fixed = 1024 + (size_t)np * W_BYTES + CL * (size_t)SLOT + SMEM_STATIC;
    if (clusters < a->u_tiles || fixed + 2 * KPS * A_BYTES > SMEM_MAX) return false;
    a->m_per_launch = clusters / a->u_tiles;
    const int fits = (int)((SMEM_MAX - fixed) / (KPS * A_BYTES)), all = (np + KPS - 1) / KPS;
    a->stages = fits < MAX_STAGES ? fits : MAX_STAGES;
    if (a->stages > all) a->stages = all < 2 ? 2 : all;
    a->smem = fixed - SMEM_STATIC + (size_t)a->stages * KPS * A_BYTES;
    return (a->m_tiles + a->m_per_launch - 1) / a->m_per_launch <= BRECUR_MAX_LAUNCHES;
}

cudaError_t wm_brecur_launch(bool f32, const void *g_map, const void *w_map, wm_brecur_args a, cudaStream_t s) {
    for (a.m0 = 0; a.m0 < a.m_tiles; a.m0 += a.m_per_launch) {
        const int mt = a.m_tiles - a.m0 < a.m_per_launch ? a.m_tiles - a.m0 : a.m_per_launch;
        cudaLaunchConfig_t lc = {};
        cudaLaunchAttribute at[2];
        set_attrs(lc, at, a.smem);
        lc.gridDim = dim3((unsigned)(CL * a.u_tiles * mt));
        lc.stream = s;
        const cudaError_t e = f32 ? cudaLaunchKernelEx(&lc, k_brecur<true>, *(const CUtensorMap *)g_map, *(const CUtensorMap *)w_map, a)
                                  : cudaLaunchKernelEx(&lc, k_brecur<false>, *(const CUtensorMap *)g_map, *(const CUtensorMap *)w_map, a);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
