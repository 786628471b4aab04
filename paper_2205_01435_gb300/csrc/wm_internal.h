// wm_internal.h -- handle layout and kernel-family launchers behind the C ABI
// of include/wm.h.  Not part of the public interface.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "wm.h"

// Device pointers of one rollout call (after host arrays were staged).
// Per-step staging of caller host arrays, for families that launch step by step: the
// family calls these around its launches on stream s so that step t's inputs arrive
// and its outputs leave on copy streams while other steps compute.
struct wm_step_stage {
    virtual cudaError_t after_init(cudaStream_t s) = 0;        // the init kernel is enqueued
    virtual cudaError_t before_step(int t, cudaStream_t s) = 0;  // before step t's first launch
    virtual cudaError_t after_step(int t, cudaStream_t s) = 0;   // after step t's last launch
    virtual bool stepping() const = 0;  // whether outputs leave step by step (after_step copies)
    virtual ~wm_step_stage() {}
};

struct wm_rollout_dev {
    wm_step_stage *stage = nullptr;  // null: the arrays are whole on the device
    int B, T;
    unsigned long long ep0;
    unsigned int t0;
    const float *z0, *h0, *c0;
    const uint8_t *done0;
    const uint32_t *mask;
    float *z_out;
    int32_t *actions;
    float *rewards;
    uint8_t *done;
    float *h_final, *c_final, *h_seq, *c_seq, *mdn_seq;
    uint8_t *comp_seq;
    const float *rt0, *mem0;   // shaped reward: predictions entering the call
    float *rt_seq, *mem_seq;   // shaped reward: predictions after each step (optional)
    float *logp_seq;           // log-prob of the action taken (optional)
    float *value_seq;          // value head V(h_{t+1}) (optional)
    const uint32_t *loc_mask;  // hierarchical action: [T, B, NX, WL] location masks (or null)
    int32_t *loc_actions;      // hierarchical action: the location taken (optional)
};

// Device pointers of one teacher-forced scoring call.
struct wm_nll_dev {
    int N, T;
    const float *z_seq;
    const int32_t *actions;
    const int32_t *lengths;
    float *nll, *h_seq, *c_seq, *mdn_seq;
    float *g_seq = nullptr;  // [T, N, 4H] gate pre-activations (tensor family, recurrence in one launch)
    // tensor family: the NLL's gradient with respect to the head outputs [T, N, M], and its bf16 copy
    float *dmd = nullptr;
    __nv_bfloat16 *dmd_op = nullptr;
};

// Weights of the stepwise (SIMT) family: fp32 values (bf16-rounded in WM_BF16).
struct wm_step_weights {
    float *Wg;   // [Z+H, 4H+A]  rows z | h; cols gates i|f|g|o then controller
    float *Wa;   // [A, 4H]      action rows of the gate matrix
    float *bg;   // [4H+A]       gate bias then controller bias
    float *Wh;   // [H, M+NR]    mixture head, reward, done (+ runtime, memory) (+ value)
    float *bh;   // [M+NR]
    float *Wp;   // [P, Z+H, A]  controller candidates (P > 1 only; else in Wg)
    float *bp;   // [P, A]
};

// Weights of the fused single-launch family: per cluster size (slot 0: 16 CTAs,
// slot 1: 8 CTAs) one bf16 image per cluster rank, laid out as in wm_fused.cu.
struct wm_fused_weights {
    void *img[2];
    size_t img_bytes[2];   // bytes per rank image
    int max_clusters[2];   // clusters of that size that can be resident at once
    int force_cluster;     // 0 = choose per call, else 8 or 16
    int ok;                // 1 if the model fits this family
};

// The fused family's small-batch member (wm_small.cu): it reads the stepwise weights;
// this records the cluster size chosen for the model and its shared-memory geometry.
struct wm_small_cfg {
    int ok;                  // 1 if the model's per-CTA columns fit a cluster's shared memory
    int cl;                  // CTAs per cluster (1, 2, 4, 8 or 16)
    int max_clusters_eb[3];  // clusters resident at once, per tile size (16, 8, 4 episodes)
    alignas(8) unsigned char geo[3][256];  // wm_small.cu's geometry record per tile size
    void *img;               // per-rank weight images (the shared-memory layout), cl of them
    size_t img_stride;       // bytes between two ranks' images
};

// Weights of the tensor-core family (bf16, K-major; orders in wm_tensor.cu).
struct wm_tc_weights {
    void *wc, *wg, *wa, *wh;  // W_c^T [P*A, Z+H], W_g^T [4H, Z+H], W_a [A, 4H], W_h^T [tiles*240, H]
    // fp32 path: the weights are the bf16 sums hi + lo; these are the lo parts (else null)
    void *wc_lo, *wg_lo, *wa_lo, *wh_lo;
    // the gate weights, action rows and bias packed again for 128-column tiles (32 units x
    // i|f|g|o per tile), for calls with few row tiles; the fp32 path's lo parts of the first two
    void *wg_n, *wa_n;
    void *wg_n_lo, *wa_n_lo;
    float *bg_n;
    float *bc, *bg, *bh;
    int dims_per_tile, n_head_tiles, rd_tile, rd_col;  // reward, done (, runtime, memory) columns
    int Zp, Hp, Ap;  // Z, H and A rounded up (zero weights) to the tiles' granularity
    int aligned;     // Zp, Hp, Ap are Z, H, A
    int sms;
    int ok;
};

// Per-kernel timing (wm_set_timing): event pairs recorded on the launching
// stream, folded into per-class totals when read.
struct wm_timer {
    struct Rec {
        int cls;
        cudaEvent_t a, b;
    };
    bool on = false;
    std::vector<Rec> pending;
    std::vector<cudaEvent_t> spare;
    double ms[WM_KERNEL_CLASSES] = {};
    long long launches[WM_KERNEL_CLASSES] = {};
};

// A canonical host copy of the weights (the layouts of wm_weights).
struct wm_host_weights {
    std::vector<float> W_lstm, b_lstm, W_mdn, b_mdn, w_rew, w_done, W_ctrl, b_ctrl, w_rt, w_mem, w_val;
    float b_rew = 0.f, b_done = 0.f, b_rt = 0.f, b_mem = 0.f, b_val = 0.f;
    wm_weights view() const {
        auto p = [](const std::vector<float> &v) { return v.empty() ? nullptr : v.data(); };
        wm_weights w{};
        w.W_lstm = p(W_lstm); w.b_lstm = p(b_lstm); w.W_mdn = p(W_mdn); w.b_mdn = p(b_mdn);
        w.w_rew = p(w_rew); w.b_rew = b_rew; w.w_done = p(w_done); w.b_done = b_done;
        w.W_ctrl = p(W_ctrl); w.b_ctrl = p(b_ctrl); w.w_rt = p(w_rt); w.b_rt = b_rt;
        w.w_mem = p(w_mem); w.b_mem = b_mem; w.w_val = p(w_val); w.b_val = b_val;
        return w;
    }
};

struct wm_handle {
    wm_config cfg;
    int device;
    int sms;                     // of the device
    int M;                       // 3 K Z
    int NR;                      // head columns after the mixture: reward, done (+ runtime,
                                 // memory when shaped) (+ value when value_head), in that order
    int P = 1, E = 1;            // controller population: candidate of episode e = (e / E) mod P
    wm_host_weights host;        // canonical host copy (repacks the fused family's images
                                 // when the controller changes)
    wm_step_weights step;
    wm_fused_weights fused;
    wm_small_cfg small;
    wm_tc_weights tc;
    void *ws = nullptr;          // workspace (grows on demand)
    size_t ws_bytes = 0;
    void *stage = nullptr;       // staging for host arrays (grows on demand)
    size_t stage_bytes = 0;
    cudaStream_t copy_in = nullptr, copy_out = nullptr;  // per-step staging copies (lazy)
    std::vector<cudaEvent_t> events;                       // per-step staging events (grows)
    int *status = nullptr;       // device status word (WM_ERR_TIMEOUT etc.)
    // tensor family, compacted rollouts: a host-mapped word the compaction kernel sets to the
    // call's sequence number once no episode is live, so that the host stops issuing steps
    mutable int *dead_host = nullptr;
    mutable int *dead_dev = nullptr;
    mutable int call_seq = 0;
    mutable std::vector<cudaEvent_t> step_events;  // the early stop's step events (lazy)
    mutable uint32_t test_wait = 0;  // wm_inject_wait_timeout: polls of the next call's injected
                                     // wait (consumed by that call's first fused / GEMM launch)
    int last_path = 0;
    mutable int last_launches = 0;   // kernels launched by the last call
    mutable wm_timer timer;
    std::string err;
    // the training step (wm_backward.cu): cuBLAS handle, copies of its GEMMs' weights (bf16 for
    // the bf16 path; W_mdn packed without the reward and done columns for the fp32 path), and its
    // workspace (all created on first use)
    void *cublas = nullptr;
    void *bw_wzh = nullptr, *bw_wm = nullptr;
    void *bw_w3 = nullptr;  // fp32 path: W_h as bf16 rows [hi | lo | hi] for the recurrence GEMM
    void *bws = nullptr;
    size_t bws_bytes = 0;
    // the one-launch recurrences: CTAs resident at once [mode][16 | 32 units][2 | 3 parts per stage]; clusters
    bool recur_ready = false, brecur_ready = false;
    int recur_ctas[3][2][2] = {};
    int brecur_clusters = 0;
};

// The current device's place in tables of per-device launch attributes.
enum { WM_MAX_DEVICES = 64 };
inline int wm_device_slot() {
    int d = 0;
    cudaGetDevice(&d);
    return d >= 0 && d < WM_MAX_DEVICES ? d : 0;
}

// Brackets the kernel launches of its scope with CUDA events on stream s when
// timing is on for h; does nothing otherwise.
class wm_ktime {
  public:
    wm_ktime(const wm_handle *h, int cls, cudaStream_t s);
    ~wm_ktime();
    wm_ktime(const wm_ktime &) = delete;
    wm_ktime &operator=(const wm_ktime &) = delete;

  private:
    wm_timer *t_;
    int cls_;
    cudaStream_t s_;
    cudaEvent_t a_ = nullptr;
};

// ---- tensor-core family (wm_tensor.cu) ----------------------------------------
int wm_tc_supported(const wm_handle *h);  // the model's sizes are multiples of the tiles'
int wm_tc_auto_ok(const wm_handle *h);    // a bf16 model it runs with its sizes padded
bool wm_tc_scores_in_one(const wm_handle *h, int N, int T);  // a scoring call's recurrence is one launch
// the operand rows [z_t | h_t] (bf16; row t N + n) that a scoring call leaves in its workspace, their
// stride and the first column of h
const __nv_bfloat16 *wm_tc_frames(const wm_handle *h, int N, int T, void *ws, int *ld, int *h_col);
// workspace of a call of B rows; T_teacher >= 0: teacher-forced scoring of T_teacher steps
// (its operand rows of all T_teacher + 1 frames), -1: a rollout
size_t wm_tc_ws(const wm_handle *h, int B, int T_teacher = -1);
cudaError_t wm_tc_pack(wm_handle *h);  // from the stepwise family's weights
void wm_tc_free(wm_handle *h);
cudaError_t wm_tc_rollout(const wm_handle *h, const wm_rollout_dev &a, void *ws, cudaStream_t s);
cudaError_t wm_tc_nll(const wm_handle *h, const wm_nll_dev &a, void *ws, cudaStream_t s);
cudaError_t wm_tc_set_controllers(wm_handle *h, int P);
// whether the tensor family can run a rollout call starting at this episode (population tiles)
int wm_tc_call_ok(const wm_handle *h, unsigned long long episode_offset);

// ---- the teacher-forced recurrence in one launch (wm_recur.cu) -----------------------
// Row tiles a CTA takes in turn, at most (more: one launch per step keeps up).
enum { RECUR_MAX_GROUPS = 4 };
struct wm_recur_args {
    int N, T, A, H, Zp, Hp, KX;
    const int32_t *act;          // [T, N]
    __nv_bfloat16 *x, *x_lo;     // [(T + 1) N, KX] operand rows of every frame (fp32 path: and lo parts)
    const __nv_bfloat16 *wa, *wa_lo;  // [A, 4Hp] action rows, and the bias, in the 128-column packing
    const float *bias;
    float *h_seq, *c_seq;        // [T, N, H] or null
    float *g_seq;                // [T, N, 4H] gate pre-activations i | f | g | o, or null
    int *count;                  // [m_tiles] zero on entry
    int *status;
    uint32_t test_wait;
    // the plan
    int units, n_tiles, m_tiles, m_groups, groups, k_steps, stages, kps;
    size_t smem;
};
// Whether (and how) N sequences run as one launch.
bool wm_recur_plan(const wm_handle *h, int mode, int N, int Hp, int KX, wm_recur_args *a);
// What the plans ask the device for, kept on the handle; before the first plan.
cudaError_t wm_recur_prepare(wm_handle *h);
cudaError_t wm_brecur_prepare(wm_handle *h);
// mode: 0 bf16, 1 bf16 with accurate nonlinearities, 2 fp32 as bf16 parts.  Tensor maps: x rows in
// boxes of 128 rows x 64, weights (128-column packing) in boxes of `units` rows x 64.
cudaError_t wm_recur_launch(int mode, const void *x_map, const void *xl_map, const void *w_map, const void *wl_map,
                            const wm_recur_args &a, cudaStream_t s);

// ---- the backward recurrence in one launch (wm_brecur.cu) ------------------------------
enum { BRECUR_MAX_LAUNCHES = 2 };  // row tiles go in as many launches as the SMs make it
struct wm_brecur_args {
    int N, T, H;
    const float *act, *cs, *dY;  // [T N, 4H] activations i | f | g | o, [T N, H] cell states, [T N, H]
    int pre;                     // act holds pre-activations
    float *dG;                   // [T N, 4H]
    __nv_bfloat16 *dGo;          // bf16 path: [T N, 4H]
    __nv_bfloat16 *parts;        // fp32 path: [2 N, 8H] rows [hi | lo] of two steps
    int *count;                  // [m_tiles] zero on entry
    int *status;
    uint32_t test_wait;          // injected wait: every CTA gives up before it issues anything
    int w_row0;                  // first row of W_h in its map
    // the plan
    int u_tiles, m_tiles, m_per_launch, m0, stages;
    size_t smem;
};
bool wm_brecur_plan(const wm_handle *h, int N, int H, wm_brecur_args *a);
// Maps: the product's operand rows (dGo, or parts) in boxes of 128 x 64; W_h's rows of units (4H gate
// columns, fp32 path: then their lo parts) in boxes of 64 x 64.
cudaError_t wm_brecur_launch(bool f32, const void *g_map, const void *w_map, wm_brecur_args a, cudaStream_t s);
// A 128-byte-swizzled map over a row-major bf16 [rows, cols] matrix (CUtensorMap *), box_rows x 64.
bool wm_tc_make_map(void *map, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows);

// ---- the fused family's small-batch member (wm_small.cu) ----------------------
cudaError_t wm_small_prepare(wm_handle *h);
cudaError_t wm_small_repack(wm_handle *h);  // after the stepwise weights changed
void wm_small_free(wm_handle *h);
int wm_small_supported(const wm_handle *h, int B);
int wm_small_cluster_size(const wm_handle *h);
cudaError_t wm_small_rollout(const wm_handle *h, const wm_rollout_dev &a, cudaStream_t s);
cudaError_t wm_small_nll(const wm_handle *h, const wm_nll_dev &a, cudaStream_t s);

// ---- the training step (wm_backward.cu) -----------------------------------------
// What the backward takes from its forward: the outputs of every row and, when the tensor family's
// one-launch recurrence ran it, the gate pre-activations and (bf16) its operand rows.
struct wm_bw_fwd {
    float *hs, *cs, *md, *nll, *G, *dMD;
    __nv_bfloat16 *dMDo;  // bf16: dMD's copy
    bool have_g, have_dmd;
    bool built;  // the weight gradients' operands X, Y are built (else: the frames, or z_seq and hs)
    const __nv_bfloat16 *frames;
    int ld, h_col;
};
// What a forward of this kernel family leaves; its workspace holds nothing that is then not read
// (of hs, md, X and Y).
wm_bw_fwd wm_bw_plan(const wm_handle *h, int N, int T, bool tensor);
size_t wm_bw_ws(const wm_handle *h, int N, int T, const wm_bw_fwd &f);
void wm_bw_carve(const wm_handle *h, int N, int T, void *base, wm_bw_fwd *f, void **tail);
cudaError_t wm_bw_prepare(wm_handle *h);
void wm_bw_free(wm_handle *h);
cudaError_t wm_bw_launch(const wm_handle *h, int N, int T, const float *z_seq, const int32_t *actions,
                         const int32_t *lengths, const wm_grads &g, const wm_bw_fwd &f, void *tail, cudaStream_t s);

// ---- discounted returns (wm_returns.cu) ----------------------------------------
cudaError_t wm_returns_launch(const wm_handle *h, int B, int T, unsigned long long ep0, float gamma,
                              int stop_at_done, const float *rewards, const uint8_t *done,
                              const float *bootstrap, float *returns, float *fitness, void *ws,
                              cudaStream_t s);
size_t wm_returns_ws(const wm_handle *h, int B);

// ---- stepwise family (wm_step.cu) -------------------------------------------
size_t wm_step_rollout_ws(const wm_handle *h, int B);
size_t wm_step_nll_ws(const wm_handle *h, int N);
cudaError_t wm_step_rollout(const wm_handle *h, const wm_rollout_dev &a, void *ws, cudaStream_t s);
cudaError_t wm_step_nll(const wm_handle *h, const wm_nll_dev &a, void *ws, cudaStream_t s);
