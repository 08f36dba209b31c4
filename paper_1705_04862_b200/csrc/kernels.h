// Host-side launchers of the PAAC kernels.  Every function enqueues work on lc.st and
// counts (and optionally times) each kernel launch through lc; none synchronises.
#pragma once
#include "common.cuh"

namespace paac {

// ---- initialisation and environment (env.cu) -----------------------------------------
void launch_init_params(LaunchCtx& lc, const NetDims& nd, uint64_t seed, float* theta);
void launch_cast_bf16(LaunchCtx& lc, const float* src, bf16* dst, size_t n);
// actions == nullptr: start states (step index 0) for every environment
void launch_env_step(LaunchCtx& lc, uint64_t seed, int n_e, const uint64_t* step_base /* device */, uint32_t t,
                     const int32_t* actions, uint32_t term_denom, uint8_t* next_frames, int8_t* rewards,
                     uint8_t* terminals, int32_t* counters /* [3][n_e] */, int pattern_actions = 0 /* > 0: the learnable
                     environment with that many actions */);

// What is left of the heads after the cluster kernel of the fully connected layer: the shares of the dot products,
// hp[parts][n_e][32], the head biases, and where logits, values, uniforms and actions go (see launch_heads_fused).
struct HeadsTail {
  const float* hp; int parts; const float* bpi; const float* bv; int A;
  float* logits; float* values; const int32_t* forced; int32_t* actions; int32_t* sampled; float* uniforms;
  HeadMode mode;
};
// the same step with the action taken inside the kernel, from the heads' partial sums
void launch_env_step_sampling(LaunchCtx& lc, uint64_t seed, int n_e, const uint64_t* step_base, uint32_t t, uint32_t term_denom,
                              uint8_t* next_frames, int8_t* rewards, uint8_t* terminals, int32_t* counters,
                              const HeadsTail& ht, int pattern_actions = 0);

// ---- external-environment mode (preprocess.cu) --------------------------------------------
// what a one-launch step of the external-environment mode does beside the network: the frame stack (newest != nullptr: the step's
// states = prev's three newest channels and the planes, four copies of the plane where fresh has the environment's bit) or
// whole states from pinned memory (states != nullptr), and actions (where sampled) and values to pinned memory, then *done = 1
struct HostStep { const uint8_t* prev; const uint8_t* newest; uint32_t fresh[3]; const uint8_t* states; int32_t* actions; float* values; volatile uint32_t* done; };
// frame stack: out = (three newest channels of prev, newest plane), or four copies of the plane where restart[e] != 0.  planes: the
// newest plane of every environment, [n][84][84] at a 16-byte aligned address, may be pinned host memory; restart: in host
// memory (nullable), read before the call returns
void launch_stack_pull(LaunchCtx& lc, const uint8_t* prev, const uint8_t* planes, const uint8_t* restart, uint8_t* out, int n);
// actions (nullable) and values of n environments to pinned host memory, then *done = 1
void launch_publish(LaunchCtx& lc, const int32_t* actions, const float* values, int n, int32_t* host_actions, float* host_values,
                    volatile uint32_t* done);

// the statistics of an update to pinned host memory, then *done = 1
void launch_publish_stats(LaunchCtx& lc, const DeviceStats* stats, DeviceStats* host_stats, volatile uint32_t* done);

void launch_advance_step(LaunchCtx& lc, uint64_t* step_base, uint32_t by);

// ---- weight gradients as split-k partial sums --------------------------------------------
// The weight-gradient kernels leave partial sums part[split][J][CO] (J = 1 for biases) in scratch regions of their own
// and note them in a GradSegments list; finish_gradients() adds them up, splits in a fixed order, into the gradient
// vector (dst[co * J + j], times scale) with one launch and empties the list.
struct GradSegment { const float* part; float* dst; int splits, J, CO; float scale; int mode, view, row_shift, co_shift; };
struct GradSegments { static constexpr int MOST = 12; GradSegment seg[MOST]; int first_group[MOST], n, total_groups; };
// in_order: one running sum over the splits (the float path's); otherwise eight interleaved ones where there are many.
// false: list full
bool add_grad_segment(GradSegments* segs, const float* part, float* dst, int splits, int J, int CO, float scale, bool in_order = false);
// sumsq_partials != nullptr: every block also leaves the sum of squares of the gradient values it wrote in
// sumsq_partials[block]; returns the number of blocks launched (at most max_blocks)
int finish_gradients(LaunchCtx& lc, GradSegments* segs, float* sumsq_partials, int max_blocks);

// ---- network on the CUDA cores (net_simt.cu) --------------------------------------------
// act[l]: stored activation of layer l for the n states, storage float (PAAC_FP32) or bf16.  Returns the number of split-k
// partial sums [split][n][F] the fully connected layer was left as in scratch (simt_scratch_floats() floats), for
// launch_simt_tail to finish; 0: the layer is complete.
int simt_forward(LaunchCtx& lc, int arch, int prec, const NetDims& nd, const float* theta,
                 const bf16* theta16, const uint8_t* frames, int n, void* const act[], float* scratch);
// scratch floats simt_backward_layer / heads_backward (n states) and simt_forward (n_fwd states) need for split-k partials
size_t simt_scratch_floats(int arch, const NetDims& nd, int n, int n_fwd);

// ---- network on the tensor cores (net_tc.cu): Nature CNN, bf16 ------------------------------
bool tc_supported(int arch, int prec);
// fc_scratch: tc_fc_scratch_floats(n) floats for the split-k partial sums of the fully connected layer
size_t tc_fc_scratch_floats(int n);
// with fc_splits != nullptr the end of the fully connected layer is shared with launch_heads_fused: either the layer
// is left as *fc_splits > 0 split-k partial sums in fc_scratch (part[split][n][512]) for that kernel to finish, or
// (*fc_splits == 0) the layer is complete and fc_scratch holds the head dot products in *head_parts shares,
// hp[parts][n][32], which that call only has to add up (see sum_head_parts)
void tc_forward(LaunchCtx& lc, int arch, const NetDims& nd, const float* theta, const bf16* theta16, const bf16* images,
                const uint8_t* frames, int n, void* const act[], float* fc_scratch, uint32_t* error_word,
                int* fc_splits = nullptr, int* head_parts = nullptr);
// transposed / regrouped bf16 weight images the backward contractions read (refreshed after every
// parameter change), and the data-gradient kernels that use them
size_t tc_weight_image_elems();
// (a first-layer weight whose fp16 image would overflow raises DEV_ERR_RANGE in *error_word)
void tc_relayout_weights(LaunchCtx& lc, const NetDims& nd, const bf16* theta16, bf16* images, uint32_t* error_word);
// one block waits at most max_polls polls on a barrier nobody signals, then records the time-out in *error_word
void launch_wait_probe(LaunchCtx& lc, uint32_t max_polls, uint32_t* error_word);
void tc_backward_dgrad_fc(LaunchCtx& lc, const bf16* images, int n, void* const act[], void* const gact[], uint32_t* err);
void tc_backward_dgrad_conv3(LaunchCtx& lc, const bf16* images, int n, void* const act[], void* const gact[], uint32_t* err);
// out_scale: power of two the gradient handed to the first layer is stored with (tc_conv1_grad_scale() when that
// layer's weight gradient runs on the tensor cores, which expects it so; 1 otherwise)
void tc_backward_dgrad_conv2(LaunchCtx& lc, const bf16* images, int n, void* const act[], void* const gact[], uint32_t* err,
                             float out_scale);
float tc_conv1_grad_scale();
// weight + bias gradients of one layer (0 = conv1 .. 3 = fc) as partial sums in the layer's own region of a scratch of
// tc_scratch_floats(B) floats, noted in the GradSegments list
size_t tc_scratch_floats(int n);
// the same data gradient followed by the first layer's weight gradient, alternating over `chunks` (at most
// TC_MAX_UPDATE_CHUNKS) groups of states; notes the weight gradient's partial sums in *segs
constexpr int TC_MAX_UPDATE_CHUNKS = 4;
void tc_backward_conv2d_conv1w_chunked(LaunchCtx& lc, const NetDims& nd, const bf16* images, const uint8_t* frames, int n,
                                       void* const act[], void* const gact[], float* grad, float* scratch, int chunks,
                                       GradSegments* segs, uint32_t* err);
void tc_backward_wgrad(LaunchCtx& lc, const NetDims& nd, const uint8_t* frames, int n, void* const act[],
                       void* const gact[], float* grad, float* scratch, int layer, GradSegments* segs, uint32_t* err);
// both heads in one kernel: gradient at the fc pre-activation into g_fc, the heads' parameter gradients as one more
// set of partial sums for finish_gradients()
bool tc_heads_backward_supported(const NetDims& nd);
void tc_heads_backward(LaunchCtx& lc, const NetDims& nd, const bf16* theta16, const bf16* h, int n, const float* dz,
                       const float* dV, bf16* g_fc, float* grad, float* scratch, GradSegments* segs);
// single layers of the CUDA-core backward pass (the tensor-core update mixes them in where it has no
// kernel of its own yet)
void simt_backward_layer(LaunchCtx& lc, int arch, int prec, const NetDims& nd, const float* theta, const bf16* theta16,
                         const uint8_t* frames, int n, void* const act[], void* const gact[], float* grad,
                         float* scratch, GradSegments* segs, int layer, bool wgrad, bool dgrad);

// ---- heads, sampling, returns, loss gradient (heads.cu) -----------------------------------
// The end of a forward pass on the CUDA cores (see simt_forward): logits / values of n states from the fully connected
// layer's partial sums (splits > 0; h is then written too) or from h; if actions != nullptr also samples; with `env` (and
// sampling) also steps the synthetic environments with the sampled actions.  advance_step: as in launch_heads_fused.
struct EnvStepArgs {
  uint32_t term_denom; uint8_t* next_frames; int8_t* rewards; uint8_t* terminals; int32_t* counters; int pattern_actions;
};
void launch_simt_tail(LaunchCtx& lc, int prec, const NetDims& nd, const float* theta, const bf16* theta16, const float* part, int splits,
                      void* h, int n, float* logits, float* values, uint64_t seed, const uint64_t* step_base, uint32_t t,
                      const int32_t* forced, int32_t* actions, int32_t* sampled /* action before forcing */, float* uniforms,
                      HeadMode mode, const EnvStepArgs* env, uint64_t* advance_step, uint32_t advance_by);
// the same for the tensor-core path, which leaves the fully connected layer as split-k partial sums
// part[split][n][F]: finishes h (sum, bias, ReLU, bf16) into h_out on the way
bool heads_fused_supported(const NetDims& nd);
void launch_heads_fused(LaunchCtx& lc, const NetDims& nd, const float* theta, const bf16* theta16, const float* part,
                        int splits, bf16* h_out, int n, float* logits, float* values, uint64_t seed,
                        const uint64_t* step_base, uint32_t t, const int32_t* forced, int32_t* actions, int32_t* sampled,
                        float* uniforms, HeadMode mode, uint64_t* advance_step = nullptr, uint32_t advance_by = 0, int parts = 2);
// advance_step (only honoured with splits == 0, only valid without sampling): the kernel also adds advance_by to the
// environments' step index, which saves the rollout its last launch
// n-step returns and advantages, the loss gradient at the heads and the loss statistics, in one launch
// mode.algo == PAAC_ALGO_NSTEP_Q: the loss is value_coef * (R - Q(s, a))^2 instead (dV = 0, no policy or entropy term)
void launch_returns_head_grad(LaunchCtx& lc, HeadMode mode, int n_e, int t_max, int A, float gamma, float beta, float value_coef,
                              const int8_t* rewards, const uint8_t* terminals, const float* logits, const float* values,
                              const int32_t* actions, float* R, float* adv, float* dz, float* dV,
                              float* loss_terms /* [3][B] */, DeviceStats* stats);
// gradient of the two heads' parameters and of the fc pre-activation
void heads_backward(LaunchCtx& lc, int prec, const NetDims& nd, const float* theta,
                    const bf16* theta16, const void* h, int n, const float* dz, const float* dV, void* gact_fc,
                    float* grad, float* scratch, GradSegments* segs);

// ---- all forward passes of a rollout in one launch, small batches of the smaller network (rollout_small.cu) ----------
bool rollout_small_supported(const LaunchCtx& lc, int arch, int prec, int n);      // sizes, and that all its blocks are resident
// what the blocks hand each other, of 16 bytes; all zero, like the two counters of SmallRollout::sync, before the first launch and
// after a device error
size_t rollout_small_words(int n);
constexpr uint32_t WORD_POLLS = 2000000u;       // a healthy wait of the one-launch rollouts ends within microseconds
struct SmallRollout {
  int n, steps, sample_steps; uint32_t t0;      // passes over slots t0 .. t0 + steps - 1; the first sample_steps sample an action
  bool step_env;                                // ... and step the synthetic environments with it (env)
  const uint8_t* frames; size_t frame_step;     // states of slot t0, bytes from one slot to the next
  void* const* act;                             // stored activations of slot t0, by layer
  void* words; uint32_t* sync;                  // rollout_small_words() or rollout_tc_words()
  float *logits, *values, *uniforms; int32_t *actions, *sampled; const int32_t* forced;      // of slot t0
  uint64_t seed; uint64_t* step_base; uint32_t advance;      // > 0: added to the step index at the end
  HostStep host;
  HeadMode mode; EnvStepArgs env;               // env.next_frames: the state after the last step; rewards, terminals of slot t0
  uint32_t* error_word; uint32_t polls;         // after which a wait gives up
};
void launch_rollout_small(LaunchCtx& lc, int prec, const NetDims& nd, const float* theta, const bf16* theta16, const SmallRollout& r);

// ---- the same for the larger network in bf16 (rollout_tc.cu) ----------
bool rollout_tc_supported(int n, int n_actions);
size_t rollout_tc_words(int n);
void launch_rollout_tc(LaunchCtx& lc, const NetDims& nd, const float* theta, const bf16* theta16, const bf16* images, const SmallRollout& r);
// what that file shares with the layer-by-layer path: the first layer's fp16 weights in `images`, the scale of their sums, and
// the number of slices of K that path adds up for n states
const void* tc_conv1_weights(const bf16* images);
float tc_conv1_scale();
int tc_fc_slices(int n);

// ---- optimiser (optim.cu) -------------------------------------------------------------------
constexpr int NORM_BLOCKS = 1184;
void launch_clip_rmsprop(LaunchCtx& lc, size_t P, float* theta, float* rms, const float* grad,
                         bf16* theta16 /* nullable */, float lr, float rho, float eps, float clip,
                         const float* norm_partials /* [0..ready_partials) hold the squared norm */, DeviceStats* stats, int ready_partials);
// the same for the larger network in bf16, with the regrouped weight images (tc_weight_images()) written from the new parameters
struct WeightImages {
  uint16_t *w1_b, *w2_d, *w3_d, *wfc_t;
  size_t w1_end, w2_off, w3_off, fc_off;        // elements of the parameter vector
  float w1_scale;
  uint32_t* error_word;
};
WeightImages tc_weight_images(const NetDims& nd, bf16* images, uint32_t* error_word);
void launch_clip_rmsprop_images(LaunchCtx& lc, size_t P, float* theta, float* rms, const float* grad, bf16* theta16, const WeightImages& img, float lr,
                                float rho, float eps, float clip, const float* norm_partials, DeviceStats* stats, int ready_partials);

}  // namespace paac
