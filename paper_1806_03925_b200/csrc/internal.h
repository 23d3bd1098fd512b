// Host-side internals of libgear: the ctx, the workspace plan and the launch functions each .cu exports.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/gear.h"
#include "common.cuh"

namespace gear {

constexpr int EXP_TILE = 8192;     // entries of the timestamp table per block of the expiry scan's write pass
constexpr int EXP_MARK_TILE = 2048; // ... and per block (and per count) of its mark pass
constexpr int MAX_LAYERS = 2;

// Byte offsets into the caller's workspace.  Everything is 256-byte aligned.
struct WsPlan {
    size_t state;                       // DevState
    // the head's matrices: bf16 (bf16 heads) or three bf16 planes of an fp32 matrix, one behind the other (fp32 heads)
    size_t x;                           // [max_batch][d_in]      head input
    size_t h[MAX_LAYERS];               // [max_batch][hidden[l]] post-ReLU activations
    size_t da[MAX_LAYERS];              // [max_batch][hidden[l]] gradient at the pre-activation
    size_t xf[MAX_LAYERS];              // fp32 head: the inputs of its layers (head input, lower hidden activations) in fp32
    size_t loss_part;                   // [loss_slots] fp32 per-block partial losses
    size_t head_grad;                   // fp32 head: the parameters' gradient, when the caller's array is not 16-byte aligned
    size_t wb[MAX_LAYERS];              // W_l as [in][out]
    size_t wbt[MAX_LAYERS];             // W_l as [out][in]
    // four sets of sort buffers: user IDs, URL IDs (max_batch each), image IDs (max_nnz), ready queue (ready_cap)
    size_t sort_keys[4][2], sort_vals[4][2];
    size_t sort_hist[4], sort_tot[4];
    int64_t sort_n[4];
    size_t tile_cnt;                    // [plan tiles + 1] uint2 per-tile (groups, complete) counts, then their totals
    size_t plan_sections;               // 64-bit counts per section of the accumulate plan
    size_t grp_rec;                     // [max_nnz] uint4 group records (start | first flag, image ID, queue slot, held rows)
    size_t blk_first;                   // [acc_max_spans] uint32: first group that starts in each span of sorted positions
    size_t run_end;                     // [max_nnz] uint32: at the first position of an image's run, one past its last
    size_t pmeta;                       // [max_nnz] int2: source row and scale (fp32 bits) of every sorted position
    size_t q_id;                        // [ready_cap] int32
    size_t q_avg;                       // [ready_cap][dfv_dim] fp32
    size_t emb_gsum[2];                 // [max_batch][emb_dim] fp32 per table: summed gradient of every distinct ID of the
                                        // batch, in the row of the sorted position where the ID's run starts (Adam only)
    size_t exp_bits;                    // [ceil(img_vocab / 32)] uint32 expired bitmap
    size_t exp_cnt;                     // [expiry mark tiles + 1][2] words: tile counts, two sets of section counts
    size_t cleared;                     // bytes from the start that a new ctx clears
    size_t total;
    int64_t ready_cap;
    int loss_blocks;
    int loss_slots;                // words of loss_part: most partial losses a batch can have
};

int plan_workspace(const gear_config& c, WsPlan* p);

class TmaCache;
TmaCache* new_tma_cache();
void delete_tma_cache(TmaCache* t);

struct gear_ctx_impl {
    gear_config cfg;
    gear_buffers buf;
    WsPlan ws;
    int d_in;
    int64_t n_params;
    cudaStream_t last_stream;
    // streams the calls were enqueued on (the expiry scan and the refresh may sit on streams of their own); the
    // calls that wait for the ctx's work wait for all of them
    static constexpr int MAX_STREAMS = 4;
    cudaStream_t seen_stream[MAX_STREAMS] = {};
    int n_seen = 0;
    void note_stream(cudaStream_t st) {
        for (int i = 0; i < n_seen; ++i) if (seen_stream[i] == st) return;
        if (n_seen < MAX_STREAMS) seen_stream[n_seen++] = st;
        else { cudaStreamSynchronize(seen_stream[0]); seen_stream[0] = st; }     // a fifth stream: retire the oldest
    }
    bool alive;
    TmaCache* tma;      // tensor maps of the head's products (tc_ptx.cuh)
    cudaStream_t side_stream;          // ID sorts, accumulate plan and embedding scatter, beside the gather and the head
    cudaStream_t aux_stream;           // expiry scan and weight gradients; for small batches the weights' copies as well
    cudaStream_t rank_stream = nullptr;  // a partitioned job's ranks (made on demand)
    cudaEvent_t ev[10];                // between the streams of a step (enqueue_step, gear_shard_step in api.cu)
    int64_t* h_counts;                 // two counts on their way to the caller (pinned; made on demand)
    Player player;                     // plays what a call has written down
    mutable Profiler prof;
    mutable bool scan_cut_off = false;      // a call failed: its expiry scan may have been enqueued in part
    mutable int plan_sections_dirty = 0;    // section counts a plan has added to and no reduce pass has cleared yet
    // image IDs of the last gear_forward_backward batch, already sorted (reused by gear_accumulate_dfv_grad)
    const int32_t* last_img_id;         // img_id array of that batch (the atomic mode reads it unsorted)
    bool img_sorted;
    int64_t img_sorted_n;
    mutable int img_sorted_buf;
    mutable bool img_sort_valid;        // the sort buffers still hold that batch's order (an accumulate call with
                                        // explicit IDs sorts into the same buffers)
    // accumulate plan made ahead by gear_forward_backward (valid for exactly these arguments)
    mutable bool plan_ready;
    mutable int64_t plan_n;
    mutable const int32_t* plan_src_row;
    mutable const float* plan_scale;
    mutable int acc_calls_pending;      // accumulate calls enqueued since a collect that was sure to drain the queue

    template <typename T> T* at(size_t off) const { return reinterpret_cast<T*>(static_cast<char*>(buf.workspace) + off); }
    DevState* state() const { return at<DevState>(ws.state); }
    enum { SORT_USER = 0, SORT_URL = 1, SORT_IMG = 2, SORT_READY = 3 };
    // a job over buffer set `which`; the caller fills ids / n / bits
    SortJob sort_job(int which) const {
        SortJob j{};
        j.keys[0] = at<uint32_t>(ws.sort_keys[which][0]); j.keys[1] = at<uint32_t>(ws.sort_keys[which][1]);
        j.vals[0] = at<uint32_t>(ws.sort_vals[which][0]); j.vals[1] = at<uint32_t>(ws.sort_vals[which][1]);
        j.hist = at<uint32_t>(ws.sort_hist[which]); j.tot = at<uint32_t>(ws.sort_tot[which]);
        j.sentinel = 0xffffffffu;
        j.status = &state()->status;
        j.identity_vals = 1;
        return j;
    }
    SortBatch sort_batch() const {
        SortBatch b{};
        b.barrier = &state()->barrier_arrived;
        b.err = &state()->tc_error;
        return b;
    }
};

// sort_small.cu: a cluster of eight blocks (one block up to 2048 IDs) per array of at most 32768 raw IDs, sorted into the first
// buffer pair of each job; the cluster of the last job also plans the accumulate call where plan.totals is set.
// What a plan is made from and where it goes (plan.cuh).
struct PlanArgs {
    uint2* totals; uint32_t vocab; const int32_t* cnt; uint4* grp_rec; const int32_t* src_row; const float* scale;
    int2* pmeta; uint32_t* blk_first; uint32_t* run_end; DevState* state;
    DivM div; int span;                         // log2 of the positions per span
};
bool sort_small_fits(const SortBatch& batch);
int64_t sort_small_max();
// the first launch of a hand-over that may have to sort the queue: count, capacity check, sort of up to sort_small_max() entries
cudaError_t launch_collect_sort(const gear_ctx_impl& c, const SortJob& job, int64_t cap, int64_t* d_n, cudaStream_t st);
cudaError_t launch_sort_small(const gear_ctx_impl& c, const SortBatch& batch, const PlanArgs& plan, cudaStream_t st);

// fill.cu
cudaError_t launch_fill_uniform(void* dst, int dtype, int64_t n_elems, uint64_t seed, uint64_t tag, double amp,
                                cudaStream_t st);
cudaError_t launch_fill_ts(int64_t* ts, int64_t n, uint64_t seed, int64_t expire, int64_t now, cudaStream_t st);

// What the weights' copies are made from (weights.cuh)
struct RoundArgs {
    int fan_in[MAX_LAYERS], fan_out[MAX_LAYERS];
    const float* W[MAX_LAYERS];
    __nv_bfloat16* wb[MAX_LAYERS];
    __nv_bfloat16* wbt[MAX_LAYERS];
    int tiles[MAX_LAYERS];                      // of 32 x 32 weights
    float* grad; int64_t n_grad;                // the parameters' gradient, cleared by the same launch
    float* loss;                                // empty batch only: its loss (0)
    int blocks() const { int n = 0; for (int t : tiles) n += t; return n; }
};
RoundArgs round_args(const gear_ctx_impl& c, const gear_step_out& o);

// gather.cu.  with_weights: the first blocks of the launch make the weights' copies and clear head_grad (bf16 heads).
cudaError_t launch_gather(const gear_ctx_impl& c, const gear_batch& b, const gear_step_out& o, bool with_weights, cudaStream_t st);

// head.cu: forward + backward of the head.  The weights' copies must have been made and head_grad cleared before it on its stream
// (launch_round_weights).  after_dx(arg) is called once dX is on its way.  The weight gradients go to dw_stream; if that is not the
// head's own stream it is made to wait for what they read (dw_ev: an event per layer), each as soon as its operands exist or,
// dw_last, all of them after dX.
struct HeadHooks { cudaError_t (*after_dx)(void*); void* arg; cudaStream_t dw_stream; cudaEvent_t* dw_ev; bool dw_last; };
cudaError_t launch_head(const gear_ctx_impl& c, const gear_batch& b, const gear_step_out& o, cudaStream_t st, const HeadHooks& hooks);
// the weights as the products read them, in a launch of their own; clears head_grad (all of it, also for an empty batch)
cudaError_t launch_round_weights(const gear_ctx_impl& c, const gear_step_out& o, cudaStream_t st);

// The blocks' partial losses of the batch, added up in a fixed order by a block of the product that follows the output unit (a
// block that found itself the last of the output unit's would keep everything behind it waiting for its fence, its ticket and
// the partials: about 2 us).  loss null: nothing to add up.
struct LossSum { const float* part; int n; int B; float* loss; };

// head_tc.cu: bf16 products on tcgen05 tensor cores.  epi: 0 bias+ReLU -> bf16, 1 ReLU mask -> bf16, 2 plain fp32.
// colsum (epi 1 only, may be null): colsum[n] += sum over the rows of the stored (rounded) output.
cudaError_t tc_gemm_kmajor(const gear_ctx_impl& c, const char* name, int M, int N, int K, const __nv_bfloat16* A, int64_t lda,
                           const __nv_bfloat16* W, int64_t ldw, int epi, void* out, int64_t ldo, const float* bias,
                           const __nv_bfloat16* mask, int64_t ldm, float* colsum, const LossSum& loss, cudaStream_t st);
// The top hidden layer and the output unit behind it: h = ReLU(A . W^T + bias) stays on the chip, dA gets the gradient with
// respect to its pre-activations.  N at most TC_TOP_N.  *n_part: how many partial losses it leaves.
constexpr int TC_TOP_N = 256;
struct TopArgs {
    const float* w_out; const float* b_out; const float* label;
    float* prob; float* loss_part; float* gw_out; float* gb_top; float* gb_out;
};
cudaError_t tc_gemm_top(const gear_ctx_impl& c, const char* name, int M, int N, int K, const __nv_bfloat16* A, int64_t lda,
                        const __nv_bfloat16* W, int64_t ldw, const float* bias, __nv_bfloat16* dA, const TopArgs& top, int* n_part, cudaStream_t st);
// out[M][N] (fp32) += A[K][M]^T . Bm[K][N]
cudaError_t tc_gemm_mnmajor(const gear_ctx_impl& c, const char* name, int M, int N, int K, const __nv_bfloat16* A, int64_t lda,
                            const __nv_bfloat16* Bm, int64_t ldb, float* out, int64_t ldo, cudaStream_t st);

// head_fwd.cu: H = ReLU(A W + bias), A [M][K], W [K][N] fp32; H in planes and, if Hf is given, in fp32
cudaError_t launch_fwd_f32(const gear_ctx_impl& c, const char* name, int M, int N, int K, const float* A, const float* W, const float* bias,
                           const Planes& H, float* Hf, cudaStream_t st);
// The same for the top hidden layer, N at most F32_TOP_N, with the output unit behind it (as tc_gemm_top): dA gets, in planes, the
// gradient with respect to its pre-activations.  fwd_top_fused_f32: whether that is the shorter way.
constexpr int F32_TOP_N = 256;
bool fwd_top_fused_f32(int M, int N, int K);
cudaError_t launch_fwd_top_f32(const gear_ctx_impl& c, int M, int N, int K, const float* A, const float* W, const float* bias,
                               const Planes& dA, const TopArgs& top, int* n_part, cudaStream_t st);

// head_tc3.cu: the backward products of fp32 matrices held as three bf16 planes.  With a mask (the leading plane of the
// activations) the output goes to planes, masked, and colsum[n] += its column sums; without, to out_f32.
cudaError_t tc3_gemm_kmajor(const gear_ctx_impl& c, const char* name, int M, int N, int K, const Planes& A, int64_t lda,
                            const Planes& W, int64_t ldw, const Planes& out_planes, float* out_f32, int64_t ldo,
                            const __nv_bfloat16* mask, int64_t ldm, float* colsum, const LossSum& loss, cudaStream_t st);
cudaError_t tc3_gemm_mnmajor(const gear_ctx_impl& c, const char* name, int M, int N, int K, const Planes& A, int64_t lda,
                             const Planes& Bm, int64_t ldb, float* out, int64_t ldo, cudaStream_t st);

// emb_scatter.cu
// table[id] += alpha * (sum of the dX rows of the views with that id) for the user and the URL-hash table, given the
// sorted (id, view) pairs of buffer sets SORT_USER / SORT_URL
cudaError_t launch_emb_reduce(const gear_ctx_impl& c, int buf, int32_t B, float* user_table, float* url_table,
                              const float* dX, int ldx, float alpha, cudaStream_t st);

// the same for arrivals: rows [.][ld], user gradients in columns 0 .. emb_dim, URL gradients behind them
cudaError_t launch_emb_arrivals(const gear_ctx_impl& c, int buf, int64_t n_user, int64_t n_url, float* user_table, float* url_table,
                                const float* rows, int64_t ld, float alpha, cudaStream_t st);

// dense.cu: a linear Dense Part (DFV = raw row . Wd) and Adam
struct EmbAdamTable { const uint32_t* ks; uint32_t vocab; float* table; float* m; float* v; const float* gsum; };
cudaError_t launch_dense_forward(const gear_ctx_impl& c, const float* raw, int R, const float* Wd, const int32_t* ids,
                                 int64_t n, const int64_t* d_n, float* rows, int64_t ld, cudaStream_t st);
cudaError_t launch_dense_backward(const gear_ctx_impl& c, const float* raw, int R, const int32_t* ids, const float* avg,
                                  int64_t ld_avg, int64_t n, const int64_t* d_n, float* G, cudaStream_t st);
cudaError_t launch_adam_dense(Profiler* prof, float* p, const float* g, float* m, float* v, int64_t n, int64_t t,
                              const gear_adam& cfg, cudaStream_t st);
cudaError_t launch_emb_adam_rows(const gear_ctx_impl& c, const EmbAdamTable& t0, const EmbAdamTable& t1, int32_t B,
                                 int64_t t, const gear_adam& cfg, cudaStream_t st);
// emb_scatter.cu: Adam on the embedding rows the batch touched (per-ID sums into compact buffers, then the row steps)
cudaError_t launch_emb_adam(const gear_ctx_impl& c, int buf, int32_t B, const float* dX, int ldx, const gear_adam& cfg,
                            int64_t t, float* user_m, float* user_v, float* url_m, float* url_v, cudaStream_t st);

// shard.cu: row fetch for a table shard's owner; event 5's gradient rows in materialised form
cudaError_t launch_fetch_rows(const gear_ctx_impl& c, int which, const int32_t* ids, int64_t n, void* out, cudaStream_t st);
cudaError_t launch_dfv_grad_rows(const gear_ctx_impl& c, const float* dX, const int32_t* row_view, const float* inv_n,
                                 int64_t nnz, float* out, cudaStream_t st);
// the exchange of a step with all ranks' shards on this device: table 0 user, 1 URL, 2 images; start[s]: where sender s's IDs
// begin in the concatenated list, start[world] = its length
struct ShardFetch {
    struct Table {
        const int32_t* ids; int32_t start[GEAR_MAX_LOCAL_RANKS + 1];
        const uint4* shard[GEAR_MAX_LOCAL_RANKS]; int64_t rows[GEAR_MAX_LOCAL_RANKS]; int chunks;      // 16-byte chunks of a row
        uint4* out[GEAR_MAX_LOCAL_RANKS];                                    // where sender s's rows go
    } table[3];
    int world;
    DevState* state[GEAR_MAX_LOCAL_RANKS];
};
struct ShardRoute {
    struct Table {
        const int32_t* ids; int32_t start[GEAR_MAX_LOCAL_RANKS + 1];
        int32_t* local; int32_t* src; int64_t src_stride;                    // [world][start[world]]
    } table[3];
    int world;
    int32_t* counts;                                                         // [3][world]
};
cudaError_t launch_shard_fetch(Profiler* prof, const ShardFetch& f, cudaStream_t st);
cudaError_t launch_shard_route(Profiler* prof, const ShardRoute& r, cudaStream_t st);
// every array becomes the mean of them all
struct ShardMean { float* p[GEAR_MAX_LOCAL_RANKS]; int world; int64_t n; };
cudaError_t launch_shard_mean(Profiler* prof, const ShardMean& m, cudaStream_t st);
// emb_scatter.cu: table[id] += alpha * (sum of the rows with that id), ids given explicitly (sorted here)
cudaError_t launch_apply_emb_grad(const gear_ctx_impl& c, int which, const int32_t* ids, const float* rows, int64_t ld,
                                  int64_t n, float alpha, cudaStream_t st);

// accumulate.cu
// img_id == nullptr: use the image IDs sorted by the last gear_forward_backward (buffer set SORT_IMG)
cudaError_t launch_accumulate(const gear_ctx_impl& c, const int32_t* img_id, const float* grads, int64_t ld,
                              const int32_t* src_row, const float* scale, int64_t n, cudaStream_t st);
// GEAR_ACC_ATOMIC: reductions on the accumulator rows, then one settle pass over the touched images
cudaError_t launch_accumulate_atomic(const gear_ctx_impl& c, const int32_t* img_id, const float* grads, int64_t ld,
                                     const int32_t* src_row, const float* scale, int64_t n, cudaStream_t st);
// steps 2-4 of the sorted accumulate for the batch just sorted by gear_forward_backward, ahead of the accumulate call
cudaError_t launch_accumulate_plan_ahead(const gear_ctx_impl& c, int64_t n, cudaStream_t st);
// ... and where its rows live and what they are scaled by, once that is known
cudaError_t launch_accumulate_resolve_ahead(const gear_ctx_impl& c, int64_t n, const int32_t* src_row, const float* scale, cudaStream_t st);
// what the plan for n rows needs; note_plan: it has been made (for the image IDs of the last batch)
PlanArgs plan_args(const gear_ctx_impl& c, int64_t n, const int32_t* src_row, const float* scale);
void note_plan(const gear_ctx_impl& c, int64_t n, const int32_t* src_row, const float* scale);
cudaError_t launch_collect_ready(const gear_ctx_impl& c, int32_t* ids, int32_t* seq, float* avg, int64_t cap,
                                 int64_t* d_n, cudaStream_t st);
// accumulate followed by the hand-over; averages bypass the queue when the host knows it to be empty and cap >= n
cudaError_t launch_accumulate_collect(const gear_ctx_impl& c, const int32_t* img_id, const float* grads, int64_t ld,
                                      const int32_t* src_row, const float* scale, int64_t n, int32_t* ids, int32_t* seq,
                                      float* avg, int64_t cap, int64_t* d_n, cudaStream_t st);

// expiry.cu
cudaError_t launch_refresh_dfv(const gear_ctx_impl& c, const int32_t* ids, const float* rows, int64_t ld, int64_t n,
                               const int64_t* d_n, int64_t now, cudaStream_t st);
cudaError_t launch_collect_expired(const gear_ctx_impl& c, int64_t now, int restamp, int32_t* ids, int64_t cap,
                                   int64_t* d_n, cudaStream_t st);

}  // namespace gear
