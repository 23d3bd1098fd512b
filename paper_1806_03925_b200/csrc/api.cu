// The C ABI of libgear (see include/gear.h): argument validation, workspace planning and the
// order in which the kernels of each call are enqueued.  No device memory is allocated here.
#include <cstdio>
#include <cstring>
#include <new>

#include "common.cuh"
#include "internal.h"

namespace gear {

static thread_local char g_last_error[256] = "";

static int cuda_fail(cudaError_t e, const char* where) {
    snprintf(g_last_error, sizeof(g_last_error), "%s: %s", where, cudaGetErrorString(e));
    return GEAR_ERR_CUDA;
}
static int arg_fail(const char* what) {
    snprintf(g_last_error, sizeof(g_last_error), "bad argument: %s", what);
    return GEAR_ERR_ARG;
}

static int validate_config(const gear_config& c) {
    const int64_t vmax = 2147483646ll;
    if (c.user_vocab < 1 || c.user_vocab > vmax || c.url_vocab < 1 || c.url_vocab > vmax || c.img_vocab < 1 ||
        c.img_vocab > vmax)
        return arg_fail("vocabulary sizes must be in [1, 2^31 - 2]");
    if (c.emb_dim < 4 || c.emb_dim % 4 || c.emb_dim > 1024) return arg_fail("emb_dim: multiple of 4 in [4, 1024]");
    if (c.dfv_dim < 8 || c.dfv_dim % 8 || c.dfv_dim > 1024) return arg_fail("dfv_dim: multiple of 8 in [8, 1024]");
    if (c.dfv_dtype != GEAR_F32 && c.dfv_dtype != GEAR_BF16) return arg_fail("dfv_dtype");
    if (c.head_dtype != GEAR_F32 && c.head_dtype != GEAR_BF16) return arg_fail("head_dtype");
    if (c.n_hidden < 1 || c.n_hidden > MAX_LAYERS) return arg_fail("n_hidden must be 1 or 2");
    for (int l = 0; l < c.n_hidden; ++l) {
        const int mult = c.head_dtype == GEAR_BF16 ? 64 : 8;
        if (c.hidden[l] < mult || c.hidden[l] % mult || c.hidden[l] > 1024)
            return arg_fail("hidden widths: multiples of 8 (fp32 head) or 64 (bf16 head), at most 1024");
    }
    if (c.M < 1) return arg_fail("M >= 1");
    if (c.expire < 0) return arg_fail("expire >= 0");
    if (c.max_batch < 1 || c.max_batch > (1 << 30) - 1) return arg_fail("max_batch in [1, 2^30 - 1]");
    const int64_t nmax = (1ll << 30) - 1;         // element counts of the key sort fit 30 bits
    if (c.max_nnz < 1 || c.max_nnz > nmax) return arg_fail("max_nnz in [1, 2^30 - 1]");
    if (c.ready_cap < 0 || c.ready_cap > nmax) return arg_fail("ready_cap in [0, 2^30 - 1]");
    if (c.accum_mode != GEAR_ACC_SORT && c.accum_mode != GEAR_ACC_ATOMIC) return arg_fail("accum_mode");
    if (c.accum_mode == GEAR_ACC_ATOMIC && c.M >= (1 << 29)) return arg_fail("GEAR_ACC_ATOMIC needs M < 2^29");
    if (c.fast_dim < 0 || c.fast_dim % 8 || c.fast_dim > 4096) return arg_fail("fast_dim: multiple of 8 in [0, 4096]");
    return GEAR_OK;
}

static int64_t param_count(const gear_config& c) {
    int64_t n = 0, fan = 2 * c.emb_dim + c.dfv_dim + c.fast_dim;
    for (int l = 0; l < c.n_hidden; ++l) { n += fan * c.hidden[l] + c.hidden[l]; fan = c.hidden[l]; }
    return n + fan + 1;
}

static int64_t plan_section_count(int64_t max_nnz) { return ceil_div(ceil_div(max_nnz, 1024), 64) + 1; }

int plan_workspace(const gear_config& c, WsPlan* p) {
    memset(p, 0, sizeof(*p));
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t at = off; off = align_up(off + bytes, 256); return at; };
    const size_t hsz = c.head_dtype == GEAR_BF16 ? 2 : 6;      // three bf16 planes per fp32 value
    const int d_in = 2 * c.emb_dim + c.dfv_dim + c.fast_dim;
    const size_t B = (size_t)c.max_batch;
    p->ready_cap = c.ready_cap > 0 ? c.ready_cap : c.max_nnz;
    p->loss_blocks = (int)ceil_div(c.max_batch, 8);
    if (p->loss_blocks > 2 * sm_count()) p->loss_blocks = 2 * sm_count();   // two resident blocks of the output-unit kernel per SM

    // an fp32 head's top layer leaves one per block, up to four resident blocks per SM
    p->loss_slots = c.head_dtype == GEAR_F32 && ceil_div(c.max_batch, 8) > p->loss_blocks ? (int)ceil_div(c.max_batch, 8) : p->loss_blocks;
    if (p->loss_slots > 4 * sm_count()) p->loss_slots = 4 * sm_count();

    // what a ctx starts with at zero, one behind the other
    p->state = take(sizeof(DevState));
    p->plan_sections = take((size_t)plan_section_count(c.max_nnz) * 8);
    p->exp_cnt = take((size_t)(ceil_div(c.img_vocab, EXP_MARK_TILE) + 1) * sizeof(uint2));
    p->cleared = off;
    p->x = take(B * d_in * hsz);
    int fan = d_in;
    for (int l = 0; l < c.n_hidden; ++l) {
        p->h[l] = take(B * c.hidden[l] * hsz);
        p->da[l] = take(B * c.hidden[l] * hsz);
        if (c.head_dtype == GEAR_F32) p->xf[l] = take(B * fan * 4);
        p->wb[l] = take((size_t)fan * c.hidden[l] * hsz);
        p->wbt[l] = take((size_t)fan * c.hidden[l] * hsz);
        fan = c.hidden[l];
    }
    p->loss_part = take((size_t)p->loss_slots * 4);
    if (c.head_dtype == GEAR_F32) p->head_grad = take((size_t)param_count(c) * 4);
    p->sort_n[0] = p->sort_n[1] = c.max_batch;
    p->sort_n[2] = c.max_nnz;
    p->sort_n[3] = p->ready_cap;
    for (int s = 0; s < 4; ++s) {
        for (int i = 0; i < 2; ++i) {
            p->sort_keys[s][i] = take((size_t)p->sort_n[s] * 4);
            p->sort_vals[s][i] = take((size_t)p->sort_n[s] * 4);
        }
        p->sort_hist[s] = take((size_t)RS_BUCKETS * sort_max_blocks(p->sort_n[s]) * 4);
        p->sort_tot[s] = take((size_t)RS_BUCKETS * 4);
    }
    p->tile_cnt = take((size_t)(ceil_div(c.max_nnz, 1024) + 1) * sizeof(uint2));
    p->grp_rec = take((size_t)c.max_nnz * 16);
    p->pmeta = take((size_t)c.max_nnz * 8);
    p->blk_first = take((size_t)acc_max_spans(c.max_nnz) * 4);
    p->run_end = take((size_t)c.max_nnz * 4);
    p->q_id = take((size_t)p->ready_cap * 4);
    p->q_avg = take((size_t)p->ready_cap * c.dfv_dim * 4);
    p->emb_gsum[0] = take(B * c.emb_dim * 4);
    p->emb_gsum[1] = take(B * c.emb_dim * 4);
    p->exp_bits = take((size_t)ceil_div(c.img_vocab, 32) * 4);
    p->total = off;
    return GEAR_OK;
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// the ctx's own streams and the events between them (host-side driver objects, no device memory)
static void release_host_objects(gear_ctx_impl& c) {
    for (cudaEvent_t& e : c.ev) { if (e) cudaEventDestroy(e); e = nullptr; }
    if (c.side_stream) cudaStreamDestroy(c.side_stream);
    if (c.aux_stream) cudaStreamDestroy(c.aux_stream);
    if (c.rank_stream) cudaStreamDestroy(c.rank_stream);
    c.rank_stream = nullptr;
    if (c.h_counts) cudaFreeHost(c.h_counts);
    c.h_counts = nullptr;
    delete_tma_cache(c.tma);
    c.tma = nullptr;
    c.side_stream = c.aux_stream = nullptr;
}

}  // namespace gear

using namespace gear;

struct gear_ctx { gear_ctx_impl impl; };

static int check_batch(const gear_ctx_impl& c, const gear_batch& b, const gear_step_out& o) {
    if (b.B < 0 || b.B > c.cfg.max_batch) return arg_fail("B outside [0, max_batch]");
    if (b.nnz < 0 || b.nnz > c.cfg.max_nnz) return arg_fail("nnz outside [0, max_nnz]");
    if (b.B > 0 && (!b.user_id || !b.url_id || !b.img_off || !b.label)) return arg_fail("NULL batch array");
    if (b.nnz > 0 && !b.img_id) return arg_fail("NULL img_id");
    if (b.B > 0 && c.cfg.fast_dim > 0 && (!b.fast || !aligned16(b.fast))) return arg_fail("fast: needed (16-byte aligned) when fast_dim > 0");
    if (!o.loss || !o.head_grad || !o.dX) return arg_fail("loss, head_grad and dX are required outputs");
    if ((o.user_grad == nullptr) != (o.url_grad == nullptr)) return arg_fail("user_grad and url_grad: both or neither");
    if (o.adam) {
        const gear_adam& a = *o.adam;
        if (o.user_grad) return arg_fail("adam and user_grad / url_grad exclude each other");
        if (!o.user_m || !o.user_v || !o.url_m || !o.url_v) return arg_fail("adam needs the four moment tables");
        if (!aligned16(o.user_m) || !aligned16(o.user_v) || !aligned16(o.url_m) || !aligned16(o.url_v))
            return arg_fail("moment tables must be 16-byte aligned");
        if (o.adam_step < 1) return arg_fail("adam_step >= 1");
        if (!(a.beta1 >= 0.f && a.beta1 < 1.f && a.beta2 >= 0.f && a.beta2 < 1.f && a.eps >= 0.f))
            return arg_fail("adam: beta1, beta2 in [0, 1), eps >= 0");
    }
    if (c.cfg.head_dtype == GEAR_BF16 && (!aligned16(o.head_grad) || !aligned16(c.buf.head_params)))
        return arg_fail("bf16 head: head_params and head_grad must be 16-byte aligned");
    if (o.dfv_grad && (!o.row_view || !o.inv_n || !aligned16(o.dfv_grad)))
        return arg_fail("dfv_grad needs row_view and inv_n and 16-byte alignment");
    if (!aligned16(o.dX) || (o.x_debug && !aligned16(o.x_debug)) || (o.user_grad && !aligned16(o.user_grad)) ||
        (o.url_grad && !aligned16(o.url_grad)))
        return arg_fail("dX, x_debug, user_grad, url_grad must be 16-byte aligned");
    return GEAR_OK;
}
static int check_rows(const gear_ctx_impl& c, const int32_t* img_id, const float* grads, int64_t ld, int64_t n) {
    if (n < 0 || n > c.cfg.max_nnz) return arg_fail("n outside [0, max_nnz]");
    if (n == 0) return GEAR_OK;
    if (!grads) return arg_fail("NULL pointer");
    if (!img_id && (!c.img_sorted || c.img_sorted_n != n)) {
        snprintf(g_last_error, sizeof(g_last_error), "img_id == NULL needs a preceding gear_forward_backward whose nnz equals n");
        return GEAR_ERR_STATE;
    }
    if (ld < c.cfg.dfv_dim || ld % 4 || !aligned16(grads)) return arg_fail("grads rows must be 16-byte aligned, ld >= dfv_dim");
    return GEAR_OK;
}
static int check_lists(const int32_t* ids, const int32_t* seq, const float* avg, int64_t cap) {
    if (cap < 0 || (cap > 0 && (!ids || !seq || !avg))) return arg_fail("NULL output with cap > 0");
    if (avg && !aligned16(avg)) return arg_fail("avg must be 16-byte aligned");
    return GEAR_OK;
}

// Events 1, 3, 4 and, where `lists` is given, 5, 6 and the expiry scan.  Written down with three streams:
//   the caller's  weight copies, gather, the head's products in the order in which they wait for one another (dA of every
//                 layer, dX), the accumulate call's reduce pass
//   side          what depends on the batch's ID arrays alone: the key sort of the three ID arrays (the user and URL orders
//                 drive the embedding scatter, the image order the accumulate call), then, once the gather has written
//                 row_view / inv_n, the accumulate call's plan; the embedding scatter as soon as dX exists
//   aux           the expiry scan (it depends on nothing a training call produces) and, for batches whose products leave SMs
//                 idle, the weight gradients, which nothing but the caller waits for
// The caller's stream waits for the other two before the call ends.  With per-kernel timing on, everything stays on the
// caller's stream so that each kernel is timed alone.
// Where one cluster sorts and plans, it does so beside the gather from more image occurrences than one block sorts by itself on, for
// bf16 heads, whose products then no longer wait for it (see enqueue_step).
constexpr int64_t EARLY_SORT_FROM = 2048;
struct StepLists {
    int32_t* ids; int32_t* seq; float* avg; int64_t cap; int64_t* d_n;
    int32_t* expired; int64_t expired_cap; int64_t* d_expired;
    int64_t now; int restamp; bool scan_beside;
};
static cudaError_t enqueue_step(gear_ctx_impl& c, const gear_batch& b, float lr, const gear_step_out& o, const StepLists* lists, cudaStream_t st) {
    c.img_sorted = false;
    c.img_sort_valid = false;
    c.plan_ready = false;
    enum { EV_FORK, EV_JOIN, EV_GATHER, EV_DX, EV_PLAN, EV_AUX };
    const bool apart = !c.prof.on || c.prof.keep_streams;
    const bool forked = apart && b.B > 0;
    const bool scan_beside = lists && apart && lists->scan_beside;
    const bool sorted_mode = c.cfg.accum_mode == GEAR_ACC_SORT;
    // Weight gradients go to a stream of their own: beside the other products while a product of the widest layer does not fill
    // the GPU by itself, else after dX, beside the store, which waits for memory where they wait for the tensor cores (65 k
    // views: step 386 -> 376 us, 32 k views fp32: 329 -> 327).
    int widest = c.d_in;
    for (int l = 0; l < c.cfg.n_hidden; ++l) widest = widest < c.cfg.hidden[l] ? c.cfg.hidden[l] : widest;
    const bool dw_beside = forked && ceil_div(b.B, 128) * ceil_div(widest, 128) <= sm_count();
    const cudaStream_t side = forked ? c.side_stream : st, aux = forked || scan_beside ? c.aux_stream : st;
    cudaError_t e = cudaSuccess;
#define GEAR_TRY(x) do { e = (x); if (e != cudaSuccess) return e; } while (0)
    if (forked || scan_beside) {
        GEAR_TRY(enqueue_record(c.ev[EV_FORK], st));
        if (forked) GEAR_TRY(enqueue_wait(side, c.ev[EV_FORK]));
        if (scan_beside) GEAR_TRY(enqueue_wait(aux, c.ev[EV_FORK]));
    }
    auto scan = [&](cudaStream_t where) {
        return launch_collect_expired(c, lists->now, lists->restamp, lists->expired, lists->expired_cap, lists->d_expired, where);
    };
    // The weights in the form the head's products read.  bf16: in the gather's launch.  (On a stream of its own a small kernel gets its
    // blocks placed only when the gather's leave room, in front of the gather it delays that by its own length, and a product
    // behind two streams starts some microseconds after the later of them.)  fp32, three planes: ahead of the gather, or, small batches,
    // which leave SMs free, beside it.
    const bool with_gather = b.B > 0 && c.cfg.head_dtype == GEAR_BF16, weights_aside = dw_beside && !with_gather;
    if (weights_aside && !scan_beside) GEAR_TRY(enqueue_wait(aux, c.ev[EV_FORK]));
    if (!with_gather) GEAR_TRY(launch_round_weights(c, o, weights_aside ? aux : st));
    if (weights_aside) GEAR_TRY(enqueue_record(c.ev[EV_AUX], aux));
    // The expiry scan reads the whole table of time stamps.  Beside the gather it slows that down; a large fp32 head's forward
    // products wait for the ALUs and leave the memory to it (32 k views: step 327 -> 316 us).  bf16 products do not (65 k views:
    // 376 us there, 386 behind the gather).
    const bool scan_late = scan_beside && forked && !dw_beside && c.cfg.head_dtype == GEAR_F32;
    if (scan_beside && !scan_late) GEAR_TRY(scan(aux));
    int sorted_buf = 0;
    bool small_sort = false;
    const bool plan = b.nnz > 0 && o.row_view && o.inv_n && sorted_mode;
    SortBatch batch = c.sort_batch();
    // a learning rate of zero moves no embedding row: nothing to sort for, nothing to scatter (a worker whose tables are
    // copies of rows that live elsewhere passes it)
    const bool scatters = lr != 0.f || o.adam || o.user_grad;
    if (b.B > 0 && scatters) {
        batch.job[0] = c.sort_job(gear_ctx_impl::SORT_USER);
        batch.job[0].ids = b.user_id; batch.job[0].sentinel = (uint32_t)c.cfg.user_vocab;
        batch.job[0].n_max = b.B; batch.job[0].bits = bits_for(c.cfg.user_vocab);
        batch.job[1] = c.sort_job(gear_ctx_impl::SORT_URL);
        batch.job[1].ids = b.url_id; batch.job[1].sentinel = (uint32_t)c.cfg.url_vocab;
        batch.job[1].n_max = b.B; batch.job[1].bits = bits_for(c.cfg.url_vocab);
        batch.n_jobs = 2;
    }
    if (b.B > 0) {
        if (b.nnz > 0 && sorted_mode) {      // the atomic mode takes the image IDs as they come
            SortJob& j = batch.job[batch.n_jobs++];
            j = c.sort_job(gear_ctx_impl::SORT_IMG);
            j.ids = b.img_id; j.sentinel = (uint32_t)c.cfg.img_vocab;
            j.n_max = b.nnz; j.bits = bits_for(c.cfg.img_vocab);
        }
        batch.name = "sort_ids";
        small_sort = batch.n_jobs > 0 && sort_small_fits(batch);
        if (batch.n_jobs > 0 && !small_sort) sorted_buf = sort_jobs(batch, side, &c.prof, &e);
        if (e != cudaSuccess) return e;
        if (b.nnz > 0) {
            c.img_sorted = true; c.img_sorted_n = b.nnz; c.img_sorted_buf = sorted_buf; c.last_img_id = b.img_id;
            c.img_sort_valid = sorted_mode;
        }
    }
    // behind the sort: the plan of the accumulate call that usually follows (which rows form which group, where every group's
    // rows and queue slot are).  Only where a row's gradient lies and its scale come from the gather (row_view, inv_n): behind a
    // multi-block sort they are put in by a launch of its own, so that the plan runs beside the gather instead of beside the
    // head's first products (65 k views: step 387 -> 381 us).  Small arrays are sorted and planned by one kernel behind the
    // gather: there the extra launch costs more than the earlier start gives (256 views +3.4 us, 1237 views fp32 34.0 / 34.3), unless
    // the head is done sooner than such a sort would be, as bf16 ones are since their weights come with the gather.  Steps of about 3
    // images a view with the sort behind the gather / beside it (us).  Below the line: 500 views, 64 units 23.4 / 25.0, 256 + 128 33.0 / 34.9,
    // 512 + 256 39.3 / 41.4.  Above it: 700 views 31.5 / 29.4, 33.9 / 34.8, 40.9 / 41.6; 1500 views 35.4 / 33.1, 37.1 / 36.4, 44.4 / 45.9;
    // 4096 views, 256 + 128 51.4 / 49.1; 7000 views 58.9 / 52.7, 59.6 / 54.0, 69.9 / 73.8; 10000 views 63.8 / 56.6, 65.8 / 59.2, 94.8 / 94.4.
    const bool early = small_sort && with_gather && b.nnz > EARLY_SORT_FROM;
    if (early) {
        GEAR_TRY(launch_sort_small(c, batch, plan ? plan_args(c, b.nnz, nullptr, nullptr) : PlanArgs{}, side));
        if (plan) note_plan(c, b.nnz, nullptr, nullptr);
    } else if (plan && forked && !small_sort) GEAR_TRY(launch_accumulate_plan_ahead(c, b.nnz, side));
    GEAR_TRY(launch_gather(c, b, o, with_gather, st));
    if (forked) GEAR_TRY(enqueue_record(c.ev[EV_GATHER], st));
    if (scan_late) {
        GEAR_TRY(enqueue_wait(aux, c.ev[EV_GATHER]));
        GEAR_TRY(scan(aux));
    }
    if (weights_aside) GEAR_TRY(enqueue_wait(st, c.ev[EV_AUX]));
    if (small_sort || (forked && plan)) {
        if (forked) GEAR_TRY(enqueue_wait(side, c.ev[EV_GATHER]));
        if (small_sort && !early) {
            GEAR_TRY(launch_sort_small(c, batch, plan ? plan_args(c, b.nnz, o.row_view, o.inv_n) : PlanArgs{}, side));
            if (plan) note_plan(c, b.nnz, o.row_view, o.inv_n);
        } else if (plan) GEAR_TRY(launch_accumulate_resolve_ahead(c, b.nnz, o.row_view, o.inv_n, side));
    }
    if (forked && lists) GEAR_TRY(enqueue_record(c.ev[EV_PLAN], side));
    // the embedding scatter: enqueued by the head as soon as dX is on its way
    struct Scatter { gear_ctx_impl* c; const gear_step_out* o; int sorted_buf; int32_t B; float lr; cudaStream_t st, side; } sc{&c, &o, sorted_buf, b.B, lr, st, side};
    auto scatter = [](void* arg) -> cudaError_t {
        Scatter& k = *static_cast<Scatter*>(arg);
        gear_ctx_impl& c = *k.c;
        const gear_step_out& o = *k.o;
        if (k.side != k.st) {
            cudaError_t e = enqueue_record(c.ev[EV_DX], k.st);
            if (e == cudaSuccess) e = enqueue_wait(k.side, c.ev[EV_DX]);
            if (e != cudaSuccess) return e;
        }
        if (o.adam)
            return launch_emb_adam(c, k.sorted_buf, k.B, o.dX, c.d_in, *o.adam, o.adam_step, o.user_m, o.user_v, o.url_m, o.url_v, k.side);
        return launch_emb_reduce(c, k.sorted_buf, k.B, o.user_grad ? o.user_grad : c.buf.user_emb, o.url_grad ? o.url_grad : c.buf.url_emb,
                                 o.dX, c.d_in, o.user_grad ? 1.0f : -k.lr, k.side);
    };
    const HeadHooks hooks{scatters ? +scatter : nullptr, &sc, forked ? aux : st, &c.ev[EV_AUX + 1], !dw_beside};
    GEAR_TRY(launch_head(c, b, o, st, hooks));
    if (o.dfv_grad && b.B > 0) GEAR_TRY(launch_dfv_grad_rows(c, o.dX, o.row_view, o.inv_n, b.nnz, o.dfv_grad, st));
    if (lists) {
        if (forked) GEAR_TRY(enqueue_wait(st, c.ev[EV_PLAN]));
        GEAR_TRY(launch_accumulate_collect(c, b.nnz > 0 ? nullptr : b.img_id, o.dX + 2 * c.cfg.emb_dim, c.d_in, o.row_view, o.inv_n, b.nnz,
                                           lists->ids, lists->seq, lists->avg, lists->cap, lists->d_n, st));
        if (!scan_beside) GEAR_TRY(scan(st));
    }
    if (forked) {
        GEAR_TRY(enqueue_record(c.ev[EV_JOIN], side));
        GEAR_TRY(enqueue_wait(st, c.ev[EV_JOIN]));
    }
    if (scan_beside || forked) {
        GEAR_TRY(enqueue_record(c.ev[EV_AUX], aux));
        GEAR_TRY(enqueue_wait(st, c.ev[EV_AUX]));
    }
#undef GEAR_TRY
    return cudaSuccess;
}

static int check_capacity(int64_t cap, int64_t n) {
    if (n <= cap) return GEAR_OK;
    snprintf(g_last_error, sizeof(g_last_error), "capacity %lld too small, %lld entries waiting", (long long)cap, (long long)n);
    return GEAR_ERR_CAPACITY;
}

// Where things lie in the staging buffer of a partitioned job (words): the five lists of the batches, the numbers of arrivals, the
// owners' results (two 64-bit counts each), and on the device only each owner's arrivals per table.
struct ShardStage {
    int64_t list[5], counts, results, local[3], src[3], host_words, words = 0;
    ShardStage(int W, int64_t max_batch, int64_t max_nnz) {
        auto take = [&](int64_t n) { const int64_t at = words; words += (n + 3) / 4 * 4; return at; };
        const int64_t cap[5] = {W * max_batch, W * max_batch, W * max_nnz, W * (max_batch + 1), W * max_batch};
        for (int t = 0; t < 5; ++t) list[t] = take(cap[t]);
        counts = take(3 * W);
        results = take(4 * W);
        host_words = words;
        for (int t = 0; t < 3; ++t) { local[t] = take(W * cap[t]); src[t] = take(W * cap[t]); }
    }
};

// both counts of a step to two pinned words (one copy where they lie side by side)
static cudaError_t enqueue_counts(void* to, const int64_t* d_n, const int64_t* d_expired, cudaStream_t st) {
    if (d_expired == d_n + 1) return enqueue_copy(to, d_n, 2 * sizeof(int64_t), st);
    cudaError_t e = enqueue_copy(to, d_n, sizeof(int64_t), st);
    return e == cudaSuccess ? enqueue_copy(static_cast<char*>(to) + sizeof(int64_t), d_expired, sizeof(int64_t), st) : e;
}
// The ctx's two pinned words.  Made when a call first waits for a count: page-locking 16 bytes takes as long as all else that
// gear_init_tables does besides filling the tables, and the contexts of a partitioned job never need them.
static cudaError_t pinned_counts(gear_ctx_impl& c) {
    return c.h_counts ? cudaSuccess : cudaHostAlloc(reinterpret_cast<void**>(&c.h_counts), 2 * sizeof(int64_t), cudaHostAllocDefault);
}

// What one owner of a partitioned job does with its arrivals.  First what their IDs alone decide: the sort (the sorted values are
// the rows' places, so no indirection is left behind it) and the accumulate plan, the expiry scan beside them.
struct Arrivals { const int32_t* ids; const int32_t* src; int64_t n; };
static cudaError_t enqueue_owner_plan(gear_ctx_impl& c, const Arrivals& user, const Arrivals& url, const Arrivals& img,
                                      const gear_step_lists& lists, int64_t now, int* sorted_buf, cudaStream_t st) {
    int64_t* d_expired = lists.d_expired ? lists.d_expired : &c.state()->pad[1];
#define GEAR_TRY(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return e_; } while (0)
    const bool apart = !c.prof.on || c.prof.keep_streams, sorted_mode = c.cfg.accum_mode == GEAR_ACC_SORT;
    const cudaStream_t aux = apart ? c.aux_stream : st;
    if (apart) {
        GEAR_TRY(enqueue_record(c.ev[0], st));
        GEAR_TRY(enqueue_wait(aux, c.ev[0]));
    }
    GEAR_TRY(launch_collect_expired(c, now, 1, lists.expired, lists.expired_cap, d_expired, aux));
    SortBatch batch = c.sort_batch();
    batch.name = "sort_ids";
    auto add = [&](const Arrivals& a, int which, int64_t vocab) {
        if (a.n == 0) return;
        SortJob& j = batch.job[batch.n_jobs++];
        j = c.sort_job(which);
        j.ids = a.ids; j.src = a.src; j.sentinel = (uint32_t)vocab; j.n_max = a.n; j.bits = bits_for(vocab);
    };
    c.img_sorted = false; c.img_sort_valid = false; c.plan_ready = false;
    add(user, gear_ctx_impl::SORT_USER, c.cfg.user_vocab);
    add(url, gear_ctx_impl::SORT_URL, c.cfg.url_vocab);
    if (sorted_mode) add(img, gear_ctx_impl::SORT_IMG, c.cfg.img_vocab);
    const bool plan = sorted_mode && img.n > 0, small_sort = batch.n_jobs > 0 && sort_small_fits(batch);
    *sorted_buf = 0;
    if (small_sort) GEAR_TRY(launch_sort_small(c, batch, plan ? plan_args(c, img.n, nullptr, nullptr) : PlanArgs{}, st));
    else if (batch.n_jobs > 0) {
        cudaError_t se;
        *sorted_buf = sort_jobs(batch, st, &c.prof, &se);
        if (se != cudaSuccess) return se;
    }
    if (plan) {
        c.img_sorted = true; c.img_sorted_n = img.n; c.img_sorted_buf = *sorted_buf; c.img_sort_valid = true; c.last_img_id = img.ids;
        if (small_sort) note_plan(c, img.n, nullptr, nullptr);
        else GEAR_TRY(launch_accumulate_plan_ahead(c, img.n, st));
    }
    if (apart) {
        GEAR_TRY(enqueue_record(c.ev[3], aux));
        GEAR_TRY(enqueue_wait(st, c.ev[3]));
    }
    return cudaSuccess;
}

// Then what their gradients do: embedding rows, gradient store and hand-over.
static cudaError_t enqueue_owner_apply(gear_ctx_impl& c, const Arrivals& user, const Arrivals& url, const Arrivals& img, int sorted_buf,
                                       const float* emb_rows, int64_t emb_ld, const float* img_rows, int64_t img_ld, float lr,
                                       const gear_step_lists& lists, void* h_counts, cudaStream_t st) {
    int64_t* d_n = lists.d_n ? lists.d_n : &c.state()->pad[0];
    int64_t* d_expired = lists.d_expired ? lists.d_expired : &c.state()->pad[1];
    const bool apart = !c.prof.on || c.prof.keep_streams, plan = c.cfg.accum_mode == GEAR_ACC_SORT && img.n > 0;
    const cudaStream_t side = apart ? c.side_stream : st;
    if (apart) {
        GEAR_TRY(enqueue_record(c.ev[1], st));
        GEAR_TRY(enqueue_wait(side, c.ev[1]));
    }
    GEAR_TRY(launch_emb_arrivals(c, sorted_buf, user.n, url.n, c.buf.user_emb, c.buf.url_emb, emb_rows, emb_ld, -lr, side));
    // (the sorted values are the source rows, so the accumulate call itself has no row indirection left)
    GEAR_TRY(launch_accumulate_collect(c, plan ? nullptr : img.ids, img_rows, img_ld, plan ? nullptr : img.src, nullptr, img.n, lists.ids,
                                       lists.seq, lists.avg, lists.cap, d_n, st));
    c.img_sorted = false; c.img_sort_valid = false;
    if (apart) {
        GEAR_TRY(enqueue_record(c.ev[2], side));
        GEAR_TRY(enqueue_wait(st, c.ev[2]));
    }
    return enqueue_counts(h_counts, d_n, d_expired, st);
#undef GEAR_TRY
}

// Waits for everything the ctx has enqueued: the stream of the training calls and, if the expiry scan went to a
// stream of its own, that one too (a call's own streams are joined to it).
static cudaError_t sync_streams(const gear_ctx_impl& c) {
    cudaError_t e = cudaStreamSynchronize(c.last_stream);
    for (int i = 0; i < c.n_seen && e == cudaSuccess; ++i)
        if (c.seen_stream[i] != c.last_stream) e = cudaStreamSynchronize(c.seen_stream[i]);
    return e;
}
// The ctx's own streams, which a call that failed may have left unjoined.
static void sync_own_streams(const gear_ctx_impl& c) {
    for (cudaStream_t s : {c.side_stream, c.aux_stream, c.rank_stream}) if (s) cudaStreamSynchronize(s);
}

// After a call that failed: nothing of it runs on a stream that the caller cannot wait for; the ctx forgets the batch whose order
// it may have been in the middle of, and whatever else the call may have left half done starts anew.
static void forget_batch(gear_ctx_impl& c) {
    sync_own_streams(c);
    c.scan_cut_off = true;
    c.acc_calls_pending = 2;                    // nothing is known of the ready queue
    c.img_sorted = false; c.img_sort_valid = false; c.plan_ready = false;
    c.plan_sections_dirty = (int)plan_section_count(c.cfg.max_nnz);
}

// Writing a call down takes host memory; that it can run out is for the caller to hear, not an exception.
template <typename Fn> static cudaError_t no_throw(Fn&& fn) {
    try { return fn(); } catch (const std::bad_alloc&) { return cudaErrorMemoryAllocation; }
}

// Writes a call down and plays it.
template <typename Fn> static int run_call(gear_ctx_impl& c, const char* where, cudaStream_t st, Fn&& enqueue) {
    c.last_stream = st;
    const cudaError_t e = no_throw([&] {
        Recording rec(c.player, st);
        const cudaError_t we = enqueue();
        return we == cudaSuccess ? rec.play(&c.prof) : we;   // (else nothing has been enqueued)
    });
    if (e == cudaSuccess) return GEAR_OK;
    forget_batch(c);
    return cuda_fail(e, where);
}

extern "C" {

const char* gear_last_error(void) { return g_last_error; }

int gear_workspace_bytes(const gear_config* cfg, size_t* out_bytes) {
    if (!cfg || !out_bytes) return arg_fail("NULL pointer");
    int rc = validate_config(*cfg);
    if (rc != GEAR_OK) return rc;
    WsPlan p;
    plan_workspace(*cfg, &p);
    *out_bytes = p.total;
    return GEAR_OK;
}

int gear_fill_uniform(void* dst, int32_t dtype, int64_t n_rows, int32_t dim, uint64_t seed, uint64_t tag, double amp,
                      void* stream) {
    if (!dst || n_rows < 0 || dim < 1 || !aligned16(dst)) return arg_fail("gear_fill_uniform");
    if (dtype != GEAR_F32 && dtype != GEAR_BF16) return arg_fail("dtype");
    cudaError_t e = launch_fill_uniform(dst, dtype, n_rows * dim, seed, tag, amp, static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? GEAR_OK : cuda_fail(e, "gear_fill_uniform");
}

int gear_init_tables(gear_ctx** out_ctx, const gear_config* cfg, const gear_buffers* buf, uint64_t seed, int fill,
                     int64_t now, void* stream) {
    if (!out_ctx || !cfg || !buf) return arg_fail("NULL pointer");
    *out_ctx = nullptr;
    int rc = validate_config(*cfg);
    if (rc != GEAR_OK) return rc;
    if (!buf->user_emb || !buf->url_emb || !buf->dfv || !buf->dfv_gsum || !buf->dfv_gcnt || !buf->dfv_ts ||
        !buf->head_params || !buf->workspace)
        return arg_fail("NULL buffer");
    if (!aligned16(buf->user_emb) || !aligned16(buf->url_emb) || !aligned16(buf->dfv) || !aligned16(buf->dfv_gsum) ||
        (reinterpret_cast<uintptr_t>(buf->workspace) & 255u))
        return arg_fail("tables must be 16-byte aligned, the workspace 256-byte aligned");
    gear_ctx* ctx = new (std::nothrow) gear_ctx;
    if (!ctx) return arg_fail("out of host memory");
    gear_ctx_impl& c = ctx->impl;
    c.cfg = *cfg;
    c.buf = *buf;
    plan_workspace(*cfg, &c.ws);
    if (buf->workspace_bytes < c.ws.total) { delete ctx; return arg_fail("workspace too small"); }
    c.d_in = 2 * cfg->emb_dim + cfg->dfv_dim + cfg->fast_dim;
    c.n_params = param_count(*cfg);
    c.alive = true;
    c.tma = new_tma_cache();
    if (!c.tma) { delete ctx; return arg_fail("out of host memory"); }
    c.img_sorted = false;
    c.img_sort_valid = false;
    c.img_sorted_n = 0;
    c.img_sorted_buf = 0;
    c.last_img_id = nullptr;
    c.acc_calls_pending = 0;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    c.last_stream = st;
    c.side_stream = c.aux_stream = nullptr;
    for (cudaEvent_t& ev : c.ev) ev = nullptr;
    c.plan_ready = false; c.plan_n = 0; c.plan_src_row = nullptr; c.plan_scale = nullptr;

    c.h_counts = nullptr;                                    // made when a count is first asked for
    cudaError_t e = cudaStreamCreateWithFlags(&c.side_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c.aux_stream, cudaStreamNonBlocking);
    for (cudaEvent_t& ev : c.ev)
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e == cudaSuccess) e = enqueue_memset(c.state(), c.ws.cleared, st);
    if (e == cudaSuccess && fill) {
        const double amp = 0.17320508075688773;   // uniform half-width for standard deviation 0.1
        e = launch_fill_uniform(buf->user_emb, GEAR_F32, cfg->user_vocab * cfg->emb_dim, seed, GEAR_TAG_USER, amp, st);
        if (e == cudaSuccess)
            e = launch_fill_uniform(buf->url_emb, GEAR_F32, cfg->url_vocab * cfg->emb_dim, seed, GEAR_TAG_URL, amp, st);
        if (e == cudaSuccess)
            e = launch_fill_uniform(buf->dfv, cfg->dfv_dtype, cfg->img_vocab * cfg->dfv_dim, seed, GEAR_TAG_DFV, amp, st);
        if (e == cudaSuccess)
            e = enqueue_memset(buf->dfv_gsum, sizeof(float) * (size_t)cfg->img_vocab * cfg->dfv_dim, st);
        if (e == cudaSuccess) e = enqueue_memset(buf->dfv_gcnt, sizeof(int32_t) * (size_t)cfg->img_vocab, st);
        if (e == cudaSuccess) e = launch_fill_ts(buf->dfv_ts, cfg->img_vocab, seed, cfg->expire, now, st);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { release_host_objects(c); delete ctx; return cuda_fail(e, "gear_init_tables"); }
    *out_ctx = ctx;
    return GEAR_OK;
}

int gear_forward_backward(gear_ctx* ctx, const gear_batch* batch, float lr, const gear_step_out* out, void* stream) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    if (!batch || !out) return arg_fail("NULL pointer");
    gear_ctx_impl& c = ctx->impl;
    if (int rc = check_batch(c, *batch, *out)) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return run_call(c, "forward_backward", st, [&] { return enqueue_step(c, *batch, lr, *out, nullptr, st); });
}

int gear_accumulate_dfv_grad(gear_ctx* ctx, const int32_t* img_id, const float* grads, int64_t ld,
                             const int32_t* src_row, const float* scale, int64_t n, void* stream) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    gear_ctx_impl& c = ctx->impl;
    if (int rc = check_rows(c, img_id, grads, ld, n)) return rc;
    if (n == 0) return GEAR_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return run_call(c, "accumulate", st, [&] {
        return c.cfg.accum_mode == GEAR_ACC_ATOMIC ? launch_accumulate_atomic(c, img_id ? img_id : c.last_img_id, grads, ld, src_row, scale, n, st)
                                                   : launch_accumulate(c, img_id, grads, ld, src_row, scale, n, st);
    });
}

static int finish_count(gear_ctx_impl& c, const int64_t* d_src, int64_t cap, int64_t* h_n, cudaStream_t st);

int gear_accumulate_collect(gear_ctx* ctx, const int32_t* img_id, const float* grads, int64_t ld, const int32_t* src_row,
                            const float* scale, int64_t n, int32_t* ids, int32_t* seq, float* avg, int64_t cap,
                            int64_t* d_n, int64_t* h_n, void* stream) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    gear_ctx_impl& c = ctx->impl;
    if (int rc = check_rows(c, img_id, grads, ld, n)) return rc;
    if (int rc = check_lists(ids, seq, avg, cap)) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int64_t* d_cnt = d_n ? d_n : &c.state()->pad[0];
    if (int rc = run_call(c, "accumulate_collect", st, [&] {
            return launch_accumulate_collect(c, img_id, grads, ld, src_row, scale, n, ids, seq, avg, cap, d_cnt, st); }))
        return rc;
    return finish_count(c, d_cnt, cap, h_n, st);
}

int gear_step(gear_ctx* ctx, const gear_batch* batch, float lr, const gear_step_out* out, const gear_step_lists* lists,
              int64_t now, int restamp, int scan_beside, int64_t* h_n, void* stream) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    if (!batch || !out || !lists) return arg_fail("NULL pointer");
    gear_ctx_impl& c = ctx->impl;
    if (int rc = check_batch(c, *batch, *out)) return rc;
    if (!out->row_view || !out->inv_n) return arg_fail("gear_step needs row_view and inv_n");
    if (batch->B == 0 && batch->nnz > 0) {          // as gear_accumulate_collect behind gear_forward_backward: there are no rows to add
        snprintf(g_last_error, sizeof(g_last_error), "image occurrences without page views");
        return GEAR_ERR_STATE;
    }
    if (int rc = check_lists(lists->ids, lists->seq, lists->avg, lists->cap)) return rc;
    if (lists->expired_cap < 0 || (lists->expired_cap > 0 && !lists->expired)) return arg_fail("NULL output with cap > 0");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const StepLists l{lists->ids, lists->seq, lists->avg, lists->cap, lists->d_n ? lists->d_n : &c.state()->pad[0],
                      lists->expired, lists->expired_cap, lists->d_expired ? lists->d_expired : &c.state()->pad[1],
                      now, restamp, scan_beside != 0};
    if (int rc = run_call(c, "step", st, [&]() -> cudaError_t {
            cudaError_t e = h_n ? pinned_counts(c) : cudaSuccess;
            if (e == cudaSuccess) e = enqueue_step(c, *batch, lr, *out, &l, st);
            return e == cudaSuccess && h_n ? enqueue_counts(c.h_counts, l.d_n, l.d_expired, st) : e;
        }))
        return rc;
    if (!h_n) return GEAR_OK;
    cudaError_t e = cudaStreamSynchronize(st);               // both counts with one wait
    if (e != cudaSuccess) return cuda_fail(e, "read counts");
    h_n[0] = c.h_counts[0]; h_n[1] = c.h_counts[1];
    if (int rc = check_capacity(l.cap, h_n[0])) return rc;
    return check_capacity(l.expired_cap, h_n[1]);
}

static int finish_count(gear_ctx_impl& c, const int64_t* d_src, int64_t cap, int64_t* h_n, cudaStream_t st) {
    if (!h_n) return GEAR_OK;
    cudaError_t e = pinned_counts(c);
    if (e == cudaSuccess) e = cudaMemcpyAsync(c.h_counts, d_src, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "read count");
    *h_n = c.h_counts[0];
    return check_capacity(cap, *h_n);
}

int gear_collect_ready(gear_ctx* ctx, int32_t* ids, int32_t* seq, float* avg, int64_t cap, int64_t* d_n, int64_t* h_n,
                       void* stream) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    gear_ctx_impl& c = ctx->impl;
    if (int rc = check_lists(ids, seq, avg, cap)) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // the count is staged in the device state so that h_n can be served even when d_n is NULL
    int64_t* d_cnt = d_n ? d_n : &c.state()->pad[0];
    if (int rc = run_call(c, "collect_ready", st, [&] { return launch_collect_ready(c, ids, seq, avg, cap, d_cnt, st); })) return rc;
    return finish_count(c, d_cnt, cap, h_n, st);
}

int gear_collect_expired(gear_ctx* ctx, int64_t now, int restamp, int32_t* ids, int64_t cap, int64_t* d_n,
                         int64_t* h_n, void* stream) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    gear_ctx_impl& c = ctx->impl;
    if (cap < 0 || (cap > 0 && !ids)) return arg_fail("NULL output with cap > 0");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    c.note_stream(st);             // may differ from the stream of the training calls: the scan shares nothing with them
    int64_t* d_cnt = d_n ? d_n : &c.state()->pad[1];
    cudaError_t e = no_throw([&] { return launch_collect_expired(c, now, restamp, ids, cap, d_cnt, st); });
    if (e != cudaSuccess) { c.scan_cut_off = true; return cuda_fail(e, "collect_expired"); }
    return finish_count(c, d_cnt, cap, h_n, st);
}

int gear_refresh_dfv(gear_ctx* ctx, const int32_t* ids, const float* rows, int64_t ld, int64_t n, const int64_t* d_n,
                     int64_t now, void* stream) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    gear_ctx_impl& c = ctx->impl;
    if (n < 0) return arg_fail("n < 0");
    if (n == 0) return GEAR_OK;
    if (!ids || !rows) return arg_fail("NULL pointer");
    if (ld < c.cfg.dfv_dim || (ld & 3) || !aligned16(rows)) return arg_fail("rows must be 16-byte aligned, ld >= dfv_dim and a multiple of 4");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    c.note_stream(st);
    cudaError_t e = no_throw([&] { return launch_refresh_dfv(c, ids, rows, ld, n, d_n, now, st); });
    if (e != cudaSuccess) return cuda_fail(e, "refresh_dfv");
    return GEAR_OK;
}

int gear_fetch_rows(gear_ctx* ctx, int32_t which, const int32_t* ids, int64_t n, void* out, void* stream) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    gear_ctx_impl& c = ctx->impl;
    if (which != GEAR_TABLE_USER && which != GEAR_TABLE_URL && which != GEAR_TABLE_DFV) return arg_fail("which");
    if (n < 0) return arg_fail("n < 0");
    if (n == 0) return GEAR_OK;
    if (!ids || !out || !aligned16(out)) return arg_fail("NULL or misaligned pointer");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    c.note_stream(st);
    cudaError_t e = no_throw([&] { return launch_fetch_rows(c, which, ids, n, out, st); });
    return e == cudaSuccess ? GEAR_OK : cuda_fail(e, "fetch_rows");
}

int gear_apply_emb_grad(gear_ctx* ctx, int32_t which, const int32_t* ids, const float* rows, int64_t ld, int64_t n, float lr,
                        void* stream) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    gear_ctx_impl& c = ctx->impl;
    if (which != GEAR_TABLE_USER && which != GEAR_TABLE_URL) return arg_fail("which: GEAR_TABLE_USER or GEAR_TABLE_URL");
    if (n < 0 || n > c.cfg.max_batch) return arg_fail("n outside [0, max_batch]");
    if (n == 0) return GEAR_OK;
    if (!ids || !rows || !aligned16(rows) || ld < c.cfg.emb_dim || (ld & 3)) return arg_fail("rows: 16-byte aligned, ld >= emb_dim, multiple of 4");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return run_call(c, "apply_emb_grad", st, [&] { return launch_apply_emb_grad(c, which, ids, rows, ld, n, -lr, st); });
}

int gear_shard_stage_words(int32_t world, int32_t max_batch, int64_t max_nnz, int64_t* words) {
    if (!words || world < 1 || world > GEAR_MAX_LOCAL_RANKS || max_batch < 1 || max_nnz < 1) return arg_fail("gear_shard_stage_words");
    *words = ShardStage(world, max_batch, max_nnz).words;
    return GEAR_OK;
}

int gear_shard_host_words(int32_t world, int32_t max_batch, int64_t max_nnz, int64_t* words) {
    if (!words || world < 1 || world > GEAR_MAX_LOCAL_RANKS || max_batch < 1 || max_nnz < 1) return arg_fail("gear_shard_host_words");
    *words = ShardStage(world, max_batch, max_nnz).host_words;
    return GEAR_OK;
}

int gear_shard_step(const gear_shard_plan* plan, const gear_host_batch* batches, float lr, int64_t now, int mean_head_grad, int64_t* counts,
                    void* stream) {
    if (!plan || !batches || !counts) return arg_fail("NULL pointer");
    const gear_shard_plan& p = *plan;
    const int W = p.world;
    if (W < 1 || W > GEAR_MAX_LOCAL_RANKS || p.max_batch < 1 || p.max_nnz < 1 || !p.owners || !p.workers || !p.host_stage || !p.stage ||
        !p.iota || !p.out || !p.lists)
        return arg_fail("gear_shard_plan");
    // ---- what the call will read and write
    gear_batch bt[GEAR_MAX_LOCAL_RANKS] = {};
    const gear_config* g0 = nullptr;
    for (int s = 0; s < W; ++s) {
        if (!p.owners[s] || !p.owners[s]->impl.alive || !p.workers[s] || !p.workers[s]->impl.alive) return GEAR_ERR_STATE;
        const gear_ctx_impl &o = p.owners[s]->impl, &w = p.workers[s]->impl;
        if (!g0) g0 = &o.cfg;
        for (const gear_config* g : {&o.cfg, &w.cfg})
            if (g->emb_dim != g0->emb_dim || g->dfv_dim != g0->dfv_dim || g->dfv_dtype != g0->dfv_dtype || g->fast_dim != 0)
                return arg_fail("the ranks' tables differ, or have a dense input of their own");
        if (w.d_in != p.workers[0]->impl.d_in || w.n_params != p.workers[0]->impl.n_params) return arg_fail("the ranks' heads differ");
        if (w.cfg.user_vocab < p.max_batch || w.cfg.url_vocab < p.max_batch || w.cfg.img_vocab < p.max_nnz) return arg_fail("a worker's tables are too small");
        const gear_host_batch& b = batches[s];
        if (b.B < 0 || b.B > p.max_batch || b.nnz < 0 || b.nnz > p.max_nnz) return arg_fail("a batch is larger than the plan's");
        if ((b.B > 0 && (!b.user_id || !b.url_id || !b.img_off || !b.label)) || (b.nnz > 0 && !b.img_id)) return arg_fail("NULL batch array");
        if (b.B == 0 && b.nnz > 0) return arg_fail("image occurrences without page views");
        const gear_step_out& out = p.out[s];
        if (!out.dfv_grad || out.dX != p.out[0].dX + (int64_t)s * p.max_batch * w.d_in ||
            out.dfv_grad != p.out[0].dfv_grad + (int64_t)s * p.max_nnz * g0->dfv_dim)
            return arg_fail("the workers' gradient rows do not lie one behind the other");
        bt[s].B = b.B; bt[s].nnz = b.nnz;
        bt[s].user_id = bt[s].url_id = bt[s].img_id = p.iota;
        bt[s].img_off = bt[s].img_id; bt[s].label = reinterpret_cast<const float*>(p.iota);      // (set below)
        if (int rc = check_batch(w, bt[s], out)) return rc;
        const gear_step_lists& l = p.lists[s];
        if (int rc = check_lists(l.ids, l.seq, l.avg, l.cap)) return rc;
        if (l.expired_cap < 0 || (l.expired_cap > 0 && !l.expired)) return arg_fail("NULL output with cap > 0");
        if ((int64_t)W * p.max_batch > o.cfg.max_batch || (int64_t)W * p.max_nnz > o.cfg.max_nnz) return arg_fail("an owner's max_batch or max_nnz is too small");
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    for (int s = 0; s < W; ++s)
        for (gear_ctx_impl* c : {&p.owners[s]->impl, &p.workers[s]->impl})
            if (e == cudaSuccess && !c->rank_stream && c != &p.owners[0]->impl)           // (owner 0 works on the caller's)
                e = cudaStreamCreateWithFlags(&c->rank_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) return cuda_fail(e, "shard_step");
    // ---- the batches: lists sender by sender in the staging buffer, one copy
    const ShardStage at(W, p.max_batch, p.max_nnz);
    ShardFetch f{};
    ShardRoute r{};
    f.world = r.world = W;
    r.counts = p.stage + at.counts;
    int64_t pos[5];
    for (int t = 0; t < 5; ++t) pos[t] = at.list[t];
    for (int s = 0; s < W; ++s) {
        const gear_host_batch& b = batches[s];
        const void* src[5] = {b.user_id, b.url_id, b.img_id, b.img_off, b.label};
        const int64_t n[5] = {b.B, b.B, b.nnz, b.B > 0 ? b.B + 1 : 0, b.B};
        bt[s].img_off = p.stage + pos[3];
        bt[s].label = reinterpret_cast<const float*>(p.stage + pos[4]);
        for (int t = 0; t < 5; ++t) {
            if (t < 3) f.table[t].start[s] = r.table[t].start[s] = (int32_t)(pos[t] - at.list[t]);
            if (n[t]) memcpy(p.host_stage + pos[t], src[t], (size_t)n[t] * 4);
            pos[t] += n[t];
        }
        const gear_ctx_impl &o = p.owners[s]->impl, &w = p.workers[s]->impl;
        f.state[s] = o.state();
        const void* shard[3] = {o.buf.user_emb, o.buf.url_emb, o.buf.dfv};
        void* rows[3] = {w.buf.user_emb, w.buf.url_emb, w.buf.dfv};
        const int64_t n_rows[3] = {o.cfg.user_vocab, o.cfg.url_vocab, o.cfg.img_vocab};
        for (int t = 0; t < 3; ++t) {
            f.table[t].shard[s] = static_cast<const uint4*>(shard[t]); f.table[t].rows[s] = n_rows[t];
            f.table[t].out[s] = static_cast<uint4*>(rows[t]);
        }
    }
    int64_t total[3];
    for (int t = 0; t < 3; ++t) {
        total[t] = pos[t] - at.list[t];
        f.table[t].ids = r.table[t].ids = p.stage + at.list[t];
        f.table[t].start[W] = r.table[t].start[W] = (int32_t)total[t];
        f.table[t].chunks = t < 2 ? g0->emb_dim / 4 : g0->dfv_dim / (g0->dfv_dtype == GEAR_BF16 ? 8 : 4);
        r.table[t].local = p.stage + at.local[t]; r.table[t].src = p.stage + at.src[t];
        r.table[t].src_stride = t < 2 ? p.max_batch : p.max_nnz;
    }
    gear_ctx_impl &w0 = p.workers[0]->impl, &o0 = p.owners[0]->impl;
    for (int s = 0; s < W; ++s) p.workers[s]->impl.last_stream = p.owners[s]->impl.last_stream = st;
    // Whatever has been enqueued is waited for, so that a caller that gives up may free the tables or use the staging buffer again
    auto fail = [&](cudaError_t err) {
        cudaStreamSynchronize(st);
        for (int s = 0; s < W; ++s)
            for (gear_ctx_impl* c : {&p.workers[s]->impl, &p.owners[s]->impl}) forget_batch(*c);
        return cuda_fail(err, "shard_step");
    };
    enum { EV_RANKS = 8, EV_ROUTED = 9 };
    // The arrivals are routed, sorted and planned on streams of their own, beside the workers' events 1 to 4: neither needs the
    // other before the gradients arrive.  (One behind the other they took 211 us for two ranks of 4096 views.)
    const bool apart = !w0.prof.on || w0.prof.keep_streams;
    auto early_of = [&](int s) { return apart ? p.workers[s]->impl.rank_stream : st; };
    const cudaStream_t early = early_of(0);
    const cudaEvent_t ev_order = o0.ev[EV_ROUTED];                        // between the caller's stream and the early ones
    auto order = [&](cudaStream_t before, cudaStream_t after) -> cudaError_t {
        if (before == after) return cudaSuccess;
        const cudaError_t re = cudaEventRecord(ev_order, before);
        return re == cudaSuccess ? cudaStreamWaitEvent(after, ev_order, 0) : re;
    };
    e = cudaMemcpyAsync(p.stage, p.host_stage, (size_t)pos[4] * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = order(st, early);
    if (e == cudaSuccess && total[0] + total[1] + total[2] > 0) e = no_throw([&] { return launch_shard_route(&w0.prof, r, early); });
    else if (e == cudaSuccess) e = cudaMemsetAsync(r.counts, 0, sizeof(int32_t) * 3 * W, early);
    if (e == cudaSuccess) e = cudaMemcpyAsync(p.host_stage + at.counts, r.counts, sizeof(int32_t) * 3 * W, cudaMemcpyDeviceToHost, early);
    if (e == cudaSuccess) e = cudaEventRecord(w0.ev[EV_ROUTED], early);
    if (e != cudaSuccess) return fail(e);
    auto stream_of = [&](int s) { return s == 0 ? st : p.owners[s]->impl.rank_stream; };
#define GEAR_TRY(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return e_; } while (0)
    // ---- events 1 to 4 on the workers, side by side
    e = no_throw([&] {
        Recording rec(w0.player, st);
        const cudaError_t we = [&]() -> cudaError_t {
            if (total[0] + total[1] + total[2] > 0) GEAR_TRY(launch_shard_fetch(&w0.prof, f, st));
            if (W > 1) GEAR_TRY(enqueue_record(w0.ev[EV_RANKS], st));
            for (int s = 1; s < W; ++s) GEAR_TRY(enqueue_wait(stream_of(s), w0.ev[EV_RANKS]));
            for (int s = 0; s < W; ++s) GEAR_TRY(enqueue_step(p.workers[s]->impl, bt[s], 0.f, p.out[s], nullptr, stream_of(s)));
            for (int s = 1; s < W; ++s) {
                GEAR_TRY(enqueue_record(p.workers[s]->impl.ev[EV_RANKS], stream_of(s)));
                GEAR_TRY(enqueue_wait(st, p.workers[s]->impl.ev[EV_RANKS]));
            }
            if (mean_head_grad && W > 1) {
                ShardMean m{};
                m.world = W; m.n = w0.n_params;
                for (int s = 0; s < W; ++s) m.p[s] = p.out[s].head_grad;
                GEAR_TRY(launch_shard_mean(&w0.prof, m, st));
            }
            return cudaSuccess;
        }();
        return we == cudaSuccess ? rec.play(&w0.prof) : we;
    });
    if (e == cudaSuccess) e = cudaEventSynchronize(w0.ev[EV_ROUTED]);
    if (e != cudaSuccess) return fail(e);
    // ---- events 4 (push), 5 and 6 at the owners, side by side
    Arrivals arrived[GEAR_MAX_LOCAL_RANKS][3];
    int sorted_buf[GEAR_MAX_LOCAL_RANKS] = {};
    for (int s = 0; s < W; ++s)
        for (int t = 0; t < 3; ++t)
            arrived[s][t] = Arrivals{r.table[t].local + s * total[t], r.table[t].src + s * total[t], (int64_t)p.host_stage[at.counts + t * W + s]};
    auto at_owners = [&](auto of, auto work) -> cudaError_t { return no_throw([&] {
        Recording rec(o0.player, of(0));
        const cudaError_t we = [&]() -> cudaError_t {
            if (W > 1) GEAR_TRY(enqueue_record(o0.ev[EV_RANKS], of(0)));
            for (int s = 0; s < W; ++s) {
                gear_ctx_impl& c = p.owners[s]->impl;
                if (s > 0) GEAR_TRY(enqueue_wait(of(s), o0.ev[EV_RANKS]));
                GEAR_TRY(work(s, c, of(s)));
                if (s > 0) {
                    GEAR_TRY(enqueue_record(c.ev[EV_ROUTED], of(s)));
                    GEAR_TRY(enqueue_wait(of(0), c.ev[EV_ROUTED]));
                }
            }
            return cudaSuccess;
        }();
        return we == cudaSuccess ? rec.play(&o0.prof) : we;
    }); };
    e = at_owners(early_of, [&](int s, gear_ctx_impl& c, cudaStream_t where) {
        return enqueue_owner_plan(c, arrived[s][0], arrived[s][1], arrived[s][2], p.lists[s], now, &sorted_buf[s], where);
    });
    if (e == cudaSuccess) e = order(early, st);
    if (e == cudaSuccess)
        e = at_owners(stream_of, [&](int s, gear_ctx_impl& c, cudaStream_t where) {
            return enqueue_owner_apply(c, arrived[s][0], arrived[s][1], arrived[s][2], sorted_buf[s], p.out[0].dX, w0.d_in, p.out[0].dfv_grad,
                                       g0->dfv_dim, lr, p.lists[s], p.host_stage + at.results + 4 * s, where);
        });
    if (e != cudaSuccess) return fail(e);
#undef GEAR_TRY
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return fail(e);
    int rc = GEAR_OK;
    for (int s = 0; s < W; ++s) {
        memcpy(counts + 2 * s, p.host_stage + at.results + 4 * s, 2 * sizeof(int64_t));
        for (int q = 0; q < 2; ++q)
            if (int bad = check_capacity(q ? p.lists[s].expired_cap : p.lists[s].cap, counts[2 * s + q])) rc = bad;
    }
    return rc;
}

int gear_dense_forward(gear_ctx* ctx, const float* raw, int32_t raw_dim, const float* Wd, const int32_t* ids, int64_t n,
                       const int64_t* d_n, float* rows, int64_t ld, void* stream) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    gear_ctx_impl& c = ctx->impl;
    if (n < 0 || raw_dim < 1) return arg_fail("n >= 0, raw_dim >= 1");
    if (n == 0) return GEAR_OK;
    if (!raw || !Wd || !ids || !rows || ld < c.cfg.dfv_dim) return arg_fail("NULL pointer or ld < dfv_dim");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    c.note_stream(st);
    cudaError_t e = no_throw([&] { return launch_dense_forward(c, raw, raw_dim, Wd, ids, n, d_n, rows, ld, st); });
    return e == cudaSuccess ? GEAR_OK : cuda_fail(e, "dense_forward");
}

int gear_dense_backward(gear_ctx* ctx, const float* raw, int32_t raw_dim, const int32_t* ids, const float* avg, int64_t n,
                        const int64_t* d_n, float* Wd_grad, void* stream) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    gear_ctx_impl& c = ctx->impl;
    if (n < 0 || raw_dim < 1) return arg_fail("n >= 0, raw_dim >= 1");
    if (n == 0) return GEAR_OK;
    if (!raw || !ids || !avg || !Wd_grad) return arg_fail("NULL pointer");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    c.note_stream(st);
    cudaError_t e = no_throw([&] { return launch_dense_backward(c, raw, raw_dim, ids, avg, c.cfg.dfv_dim, n, d_n, Wd_grad, st); });
    return e == cudaSuccess ? GEAR_OK : cuda_fail(e, "dense_backward");
}

int gear_adam_dense(float* param, const float* grad, float* m, float* v, int64_t n, int64_t t, const gear_adam* cfg,
                    void* stream) {
    if (n < 0 || t < 1 || !cfg) return arg_fail("n >= 0, t >= 1, cfg");
    if (n == 0) return GEAR_OK;
    if (!param || !grad || !m || !v) return arg_fail("NULL pointer");
    if (!(cfg->beta1 >= 0.f && cfg->beta1 < 1.f && cfg->beta2 >= 0.f && cfg->beta2 < 1.f && cfg->eps >= 0.f))
        return arg_fail("adam: beta1, beta2 in [0, 1), eps >= 0");
    cudaError_t e = no_throw([&] { return launch_adam_dense(nullptr, param, grad, m, v, n, t, *cfg, static_cast<cudaStream_t>(stream)); });
    return e == cudaSuccess ? GEAR_OK : cuda_fail(e, "adam_dense");
}

int gear_status(gear_ctx* ctx, int32_t* device_status, int64_t* pending_ready) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    gear_ctx_impl& c = ctx->impl;
    DevState h;
    memset(&h, 0, sizeof(h));
    cudaError_t e = sync_streams(c);
    if (e == cudaSuccess) e = cudaMemcpy(&h, c.state(), sizeof(DevState), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "gear_status");      // h holds nothing to look at
    if (h.tc_error != 0) h.status |= GEAR_DEV_TIMEOUT;
    if (e == cudaSuccess && h.status != 0) e = cudaMemset(c.state(), 0, 2 * sizeof(int32_t));   // status, tc_error
    if (e != cudaSuccess) return cuda_fail(e, "gear_status");
    if (device_status) *device_status = h.status;
    if (pending_ready) *pending_ready = h.q_count;
    if (h.status & GEAR_DEV_TIMEOUT) {
        snprintf(g_last_error, sizeof(g_last_error), "a bounded device wait gave up (code %d)", h.tc_error);
        return GEAR_ERR_CUDA;
    }
    if (h.status & GEAR_DEV_BAD_ID) return GEAR_ERR_BAD_ID;
    if (h.status & (GEAR_DEV_READY_OVERFLOW | GEAR_DEV_OUT_CAPACITY)) return GEAR_ERR_CAPACITY;
    if (h.status & GEAR_DEV_BAD_CSR) return GEAR_ERR_ARG;
    return GEAR_OK;
}

int gear_profile_enable(gear_ctx* ctx, int on) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    sync_streams(ctx->impl);
    ctx->impl.prof.clear();
    ctx->impl.prof.on = on != 0;
    ctx->impl.prof.keep_streams = on == 2;
    return GEAR_OK;
}

int gear_profile_timeline(gear_ctx* ctx, char* names, float* start_ms, float* stop_ms, int32_t cap, int32_t* n_out) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    if (!n_out || cap < 0 || (cap > 0 && (!names || !start_ms || !stop_ms))) return arg_fail("gear_profile_timeline");
    gear_ctx_impl& c = ctx->impl;
    cudaError_t e = sync_streams(c);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c.side_stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c.aux_stream);
    if (e != cudaSuccess) return cuda_fail(e, "gear_profile_timeline");
    int n = 0;
    for (const auto& r : c.prof.recs) {
        if (n >= cap) break;
        float a = 0.f, b = 0.f;
        e = cudaEventElapsedTime(&a, c.prof.recs[0].start, r.start);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&b, c.prof.recs[0].start, r.stop);
        if (e != cudaSuccess) return cuda_fail(e, "cudaEventElapsedTime");
        strncpy(names + 64 * n, r.name, 63);
        names[64 * n + 63] = 0;
        start_ms[n] = a; stop_ms[n] = b;
        ++n;
    }
    *n_out = n;
    c.prof.clear();
    return GEAR_OK;
}

int gear_profile_read(gear_ctx* ctx, char* names, float* total_ms, int32_t* launches, int32_t cap, int32_t* n_out) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    if (!n_out || cap < 0 || (cap > 0 && (!names || !total_ms || !launches))) return arg_fail("gear_profile_read");
    gear_ctx_impl& c = ctx->impl;
    cudaError_t e = sync_streams(c);
    if (e != cudaSuccess) return cuda_fail(e, "gear_profile_read");
    int n = 0;
    for (const auto& r : c.prof.recs) {
        float ms = 0.f;
        e = cudaEventElapsedTime(&ms, r.start, r.stop);
        if (e != cudaSuccess) return cuda_fail(e, "cudaEventElapsedTime");
        int k = 0;
        while (k < n && strncmp(names + 64 * k, r.name, 63) != 0) ++k;
        if (k == n) {
            if (n >= cap) continue;
            strncpy(names + 64 * k, r.name, 63);
            names[64 * k + 63] = 0;
            total_ms[k] = 0.f;
            launches[k] = 0;
            ++n;
        }
        total_ms[k] += ms;
        launches[k] += 1;
    }
    *n_out = n;
    c.prof.clear();
    return GEAR_OK;
}

int gear_launch_count(gear_ctx* ctx, int64_t* n_launches) {
    if (!ctx || !ctx->impl.alive) return GEAR_ERR_STATE;
    if (!n_launches) return arg_fail("NULL pointer");
    *n_launches = ctx->impl.prof.launches;
    return GEAR_OK;
}

int gear_destroy(gear_ctx* ctx) {
    if (!ctx) return GEAR_OK;
    if (!ctx->impl.alive) return GEAR_ERR_STATE;     // a ctx that failed half-way through its set-up; a destroyed
                                                     // ctx is freed memory and must not be passed in again
    sync_streams(ctx->impl);
    sync_own_streams(ctx->impl);
    release_host_objects(ctx->impl);
    ctx->impl.alive = false;
    delete ctx;
    return GEAR_OK;
}

}  // extern "C"
