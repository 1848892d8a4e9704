// api.cu -- the C ABI entry points (include/impact.h). A call works on a
// batch of builds (a single build is a batch of one): the planner (plan.cu)
// makes each build's descriptor and tables, this file lays them out with the
// batch index, the scan scratch and the per-row records in one device
// workspace, and runs the count -> scan -> emit pipeline on the caller's
// stream, directly or as a captured CUDA graph. It also holds the launch-shape
// autotuner of the FP32 walk.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <string>
#include <unordered_map>
#include <vector>

#include "../../include/impact.h"
#include "alloc.h"
#include "impact_desc.h"
#include "kernels.h"
#include "pipeline.h"
#include "plan.h"

namespace {
thread_local std::string g_last_error;
}  // namespace

namespace impact {
impact_status fail(impact_status s, const std::string &msg)
{
    g_last_error = msg;
    return s;
}
void set_last_error(const std::string &msg) { g_last_error = msg; }
}  // namespace impact


#define CK(expr)                                                                              \
    do {                                                                                      \
        cudaError_t e_ = (expr);                                                              \
        if (e_ != cudaSuccess) {                                                              \
            return fail(e_ == cudaErrorMemoryAllocation ? IMPACT_ERR_OOM : IMPACT_ERR_CUDA,   \
                        std::string(#expr) + ": " + cudaGetErrorString(e_));                 \
        }                                                                                     \
    } while (0)

namespace impact {

constexpr int kBatchMax = 1 << 16;   // builds per batch

uint64_t mix(uint64_t h, uint64_t v)
{
    for (int i = 0; i < 8; ++i) h = (h ^ ((v >> (8 * i)) & 0xff)) * 1099511628211ull;
    return h;
}

impact_status tuning_of(const impact_tuning *t, Tuning &T)
{
    T = Tuning();
    if (!t) return IMPACT_OK;
    if (t->count_warps) T.count_warps = t->count_warps;
    if (t->emit_warps) T.emit_warps = t->emit_warps;
    if (T.count_warps < 1 || T.count_warps > IMPACT_TREE_WARPS_MAX || T.emit_warps < 1 ||
        T.emit_warps > IMPACT_TREE_WARPS_MAX)
        return fail(IMPACT_ERR_ARG, "tuning: warps per block must be in [1, 8]");
    if (t->spin_limit < 0 || t->stall_row < 0 || t->fault_row < 0 || t->guard_row < 0 ||
        (t->one_pass != 0 && t->one_pass != 1))
        return fail(IMPACT_ERR_ARG,
                    "tuning: spin_limit, stall_row, fault_row and guard_row must be >= 0, "
                    "one_pass 0 or 1");
    T.one_pass = t->one_pass == 1;
    T.faults.spin_limit = t->spin_limit;
    T.faults.stall_row = t->stall_row - 1;
    T.faults.fault_row = t->fault_row - 1;
    T.faults.guard_row = t->guard_row - 1;
    return IMPACT_OK;
}

// ---------------------------------------------------------------------------
// batches
// ---------------------------------------------------------------------------


// What the passes of build q need beside those before it: item and leaf table
// numbering, shared memory.
void size_build(Batch &B, int q)
{
    const ImpactDesc &D = B.plans[q].desc;
    if (B.prec == IMPACT_FP32_SOUND) {
        B.rec_max = std::max(B.rec_max, D.rec_stride);
        for (int mode = 0; mode < 3; ++mode)
            B.work_max[mode] = std::max(B.work_max[mode], impact::walk_work_bytes(D, mode));
    }
    for (int d = 0; d < IMPACT_MAX_DIM; ++d) {
        const size_t i = (size_t)q * IMPACT_MAX_DIM + d;
        int64_t units = 0;
        if ((D.walk64 || D.share32) && d < D.n) {
            const int ipw = 32 / D.dim[d].group;
            units = (D.dim[d].n_items + ipw - 1) / ipw;
        }
        B.item_begin[i + 1] = B.item_begin[i] + units;
    }
    B.leaf_begin[q + 1] = B.leaf_begin[q] + (D.leaf_shared ? D.leaf_items : 0);
    if (D.leaf_shared) B.leaf_smem = std::max(B.leaf_smem, impact::leaf32_bytes(D));
    if (D.share32) ++B.shared32;
    if (D.walk64) {
        ++B.any64;
        B.warp64 = std::max(B.warp64, (int)impact::walk64_bytes(D));
    }
}

bool make_lean(Batch &B, int only)
{
    const int from = only < 0 ? 0 : only, to = only < 0 ? B.count() : only + 1;
    int64_t spare = 0;
    for (int q = from; q < to; ++q)
        spare += B.plans[q].leaf_bytes + (B.plans[q].desc.walk64 ? B.plans[q].item_bytes : 0);
    if (!B.walks || spare < kSpareMin) return false;
    for (int q = from; q < to; ++q) {
        Plan &P = B.plans[q];
        if (P.desc.walk64) P.item_bytes = 0;
        P.leaf_bytes = 0;
        P.desc.walk64 = P.desc.leaf_shared = P.desc.lists = 0;
    }
    B.rec_max = B.leaf_smem = B.shared32 = B.any64 = B.warp64 = 0;
    for (int &w : B.work_max) w = 0;
    for (int q = 0; q < B.count(); ++q) size_build(B, q);
    return true;
}

impact_status make_batch(const impact_request *reqs, int count, impact_precision precision,
                         const impact_tuning *tuning, Batch &B)
{
    if (!reqs) return fail(IMPACT_ERR_ARG, "null request array");
    if (count < 1 || count > kBatchMax)
        return fail(IMPACT_ERR_ARG, "request count must be in [1, 65536]");
    impact_status s = tuning_of(tuning, B.tune);
    if (s != IMPACT_OK) return s;
    B.plans.assign(count, Plan());
    B.images.assign(count, nullptr);
    B.row_begin.assign(count + 1, 0);
    B.unit_begin.assign(count + 1, 0);
    B.item_begin.assign((size_t)count * IMPACT_MAX_DIM + 1, 0);
    B.leaf_begin.assign(count + 1, 0);
    B.prec = precision;
    uint64_t h = 1469598103934665603ull;
    for (int q = 0; q < count; ++q) {
        const impact_request &r = reqs[q];
        s = impact::make_plan(r.sys, r.grid, r.inputs, r.sigma, r.cutoff, precision, B.plans[q]);
        if (s != IMPACT_OK) {
            if (count > 1) g_last_error = "request " + std::to_string(q) + ": " + g_last_error;
            return s;
        }
        const Plan &P = B.plans[q];
        B.images[q] = r.sys->dev_images;
        B.row_begin[q + 1] = B.row_begin[q] + P.rows;
        const int64_t rpw = 32 / P.desc.n;
        B.unit_begin[q + 1] = B.unit_begin[q] + (P.rows + rpw - 1) / rpw;
        B.nnz_bound = (B.nnz_bound > INT64_MAX - P.nnz_bound) ? INT64_MAX
                                                              : B.nnz_bound + P.nnz_bound;
        size_build(B, q);
        h = mix(h, P.hash);
    }
    B.rows = B.row_begin[count];
    B.units = B.unit_begin[count];
    B.hash = h;   // launch shapes change no result: they are not part of the identity
    if (precision == IMPACT_FP32_SOUND &&
        2 * (int64_t)B.rec_max + B.work_max[WALK_FUSED] > IMPACT_WALK_SMEM_MAX)
        return fail(IMPACT_ERR_ARG,
                    "the builds of this batch together need " +
                        std::to_string(2 * (int64_t)B.rec_max + B.work_max[WALK_FUSED]) +
                        " bytes of shared memory per warp, more than one warp has: "
                        "batch the widest windows separately");
    return IMPACT_OK;
}


BatchLayout batch_layout(const Batch &B)
{
    BatchLayout L;
    size_t o = 0;
    auto put = [&](size_t bytes) {
        size_t at = o;
        o = impact::align256(o + bytes);
        return at;
    };
    const int count = B.count();
    L.index = put(sizeof(BatchIndex));
    L.row_begin = put((size_t)(count + 1) * 8);
    L.unit_begin = put((size_t)(count + 1) * 8);
    L.descs = put((size_t)count * 8);
    L.recs = put((size_t)count * 8);
    L.items = put((size_t)count * 8);
    L.leafs = put((size_t)count * 8);
    L.termps = put((size_t)count * 8);
    L.item_begin = put(B.item_begin.size() * 8);
    L.leaf_begin = put(B.leaf_begin.size() * 8);
    L.tables.resize(count);
    L.tl.resize(count);
    for (int q = 0; q < count; ++q) {
        L.tl[q] = impact::table_layout(B.plans[q]);
        L.tables[q] = put(L.tl[q].total);
    }
    L.status = put(64);
    L.upload_end = L.status + 64;   // its zeros go up with the tables
    L.scan = put((size_t)impact::scan_scratch_elems(B.rows) * 8);
    L.lb = put(!B.walks                    ? 0
               : B.prec == PREC_FP32_SOUND ? (size_t)B.rows * 16
                                           : (B.any64 ? (size_t)B.rows * 24 : 0));
    L.rec.resize(count);
    L.item.resize(count);
    L.leaf.resize(count);
    L.term.resize(count);
    for (int q = 0; q < count; ++q) {
        const Plan &P = B.plans[q];
        const bool rec = B.walks && B.prec == PREC_FP32_SOUND;
        L.rec[q] = put(rec ? (size_t)P.rows * P.desc.rec_stride : 0);
        L.item[q] = put(B.walks ? (size_t)P.item_bytes : 0);
        L.term[q] = put(rec && !P.desc.share32 ? (size_t)P.rows * P.desc.n * 16 : 0);
        L.leaf[q] = put(B.walks ? (size_t)P.leaf_bytes : 0);
    }
    L.extra = put((size_t)B.extra);
    L.total = o;
    return L;
}


std::mutex g_ws_mu;
std::unordered_map<const void *, uint64_t> g_ws_tag;   // caller workspace -> batch it holds

void ws_tag(const void *ws, uint64_t h)
{
    std::lock_guard<std::mutex> lock(g_ws_mu);
    if (h) g_ws_tag[ws] = h; else g_ws_tag.erase(ws);
}

bool ws_has(const void *ws, uint64_t h)
{
    std::lock_guard<std::mutex> lock(g_ws_mu);
    auto it = g_ws_tag.find(ws);
    return it != g_ws_tag.end() && it->second == h;
}

impact_status get_work(Batch &B, const impact_csr *out, cudaStream_t st, Work &W)
{
    W.L = batch_layout(B);
    if (out && out->workspace) {
        if (out->workspace_bytes < (int64_t)W.L.total)
            return fail(IMPACT_ERR_ARG, "workspace too small: " +
                                            std::to_string(out->workspace_bytes) + " < " +
                                            std::to_string(W.L.total) + " bytes");
        if (((uintptr_t)out->workspace & 255) != 0)
            return fail(IMPACT_ERR_ARG, "workspace must be 256-byte aligned");
        W.base = (unsigned char *)out->workspace;
        W.owned = false;
        return IMPACT_OK;
    }
    cudaError_t e = dev_malloc_async(&W.base, W.L.total, st);
    if (e == cudaErrorMemoryAllocation && make_lean(B)) {
        W.L = batch_layout(B);
        e = dev_malloc_async(&W.base, W.L.total, st);
    }
    if (e != cudaSuccess)
        return fail(e == cudaErrorMemoryAllocation ? IMPACT_ERR_OOM : IMPACT_ERR_CUDA,
                    std::string("workspace: ") + cudaGetErrorString(e));
    W.owned = true;
    return IMPACT_OK;
}

impact_status release(Work &W, cudaStream_t st)
{
    unsigned char *b = W.base;
    W.base = nullptr;
    if (W.owned && b) CK(dev_free_async(b, st));
    return IMPACT_OK;
}

// Releases a library-owned workspace on every return path that did not
// release it already.
struct WorkHold {
    Work &W;
    cudaStream_t st;
    ~WorkHold() { release(W, st); }
};

// Frees the arrays of a library-owned result (stream-ordered) and clears
// them, keeping the caller's workspace fields.
void free_owned(impact_csr *out, cudaStream_t st)
{
    void *ptrs[] = {out->row_ptr, out->col, out->lo, out->up, out->sink_lo,
                    out->sink_up, out->trunc, out->row_flags};
    for (void *p : ptrs) dev_free_async(p, st);
    void *ws = out->workspace;
    int64_t wsb = out->workspace_bytes;
    memset(out, 0, sizeof(*out));
    out->workspace = ws;
    out->workspace_bytes = wsb;
}

// Copies the batch index, the descriptors, the tables and a zeroed status block
// into the workspace.
impact_status upload(const Batch &B, Work &W, cudaStream_t st)
{
    const BatchLayout &L = W.L;
    const int count = B.count();
    std::vector<unsigned char> host(L.upload_end, 0);
    BatchIndex bi;
    memset(&bi, 0, sizeof(bi));
    bi.count = count;
    bi.rows = B.rows;
    bi.units = B.units;
    bi.row_begin = (const int64_t *)(W.base + L.row_begin);
    bi.unit_begin = (const int64_t *)(W.base + L.unit_begin);
    bi.desc = (const ImpactDesc *const *)(W.base + L.descs);
    bi.rec = (unsigned char *const *)(W.base + L.recs);
    bi.next_row = W.counter();
    bi.items = (unsigned char *const *)(W.base + L.items);
    bi.terms = (unsigned char *const *)(W.base + L.termps);
    bi.leaf = (unsigned char *const *)(W.base + L.leafs);
    bi.item_units = B.item_begin.back();
    bi.item_begin = (const int64_t *)(W.base + L.item_begin);
    bi.leaf_total = B.leaf_begin.back();
    bi.leaf_begin = (const int64_t *)(W.base + L.leaf_begin);
    memcpy(host.data() + L.index, &bi, sizeof(bi));
    memcpy(host.data() + L.row_begin, B.row_begin.data(), (size_t)(count + 1) * 8);
    memcpy(host.data() + L.unit_begin, B.unit_begin.data(), (size_t)(count + 1) * 8);
    memcpy(host.data() + L.item_begin, B.item_begin.data(), B.item_begin.size() * 8);
    memcpy(host.data() + L.leaf_begin, B.leaf_begin.data(), B.leaf_begin.size() * 8);
    for (int q = 0; q < count; ++q) {
        const ImpactDesc *d = W.desc(q);
        unsigned char *r = W.base + L.rec[q], *i = W.base + L.item[q], *f = W.base + L.leaf[q],
                      *v = W.base + L.term[q];
        memcpy(host.data() + L.descs + 8 * (size_t)q, &d, 8);
        memcpy(host.data() + L.recs + 8 * (size_t)q, &r, 8);
        memcpy(host.data() + L.items + 8 * (size_t)q, &i, 8);
        memcpy(host.data() + L.leafs + 8 * (size_t)q, &f, 8);
        memcpy(host.data() + L.termps + 8 * (size_t)q, &v, 8);
        impact::pack_tables(B.plans[q], host.data() + L.tables[q], W.base + L.tables[q],
                            B.images[q]);
    }
    // pageable source: returns once the bytes are staged, so `host` may go
    CK(cudaMemcpyAsync(W.base, host.data(), host.size(), cudaMemcpyHostToDevice, st));
    return IMPACT_OK;
}

void configure_pool_once()
{
    static std::once_flag once;
    std::call_once(once, [] {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return;
        cudaMemPool_t pool;
        if (cudaDeviceGetDefaultMemPool(&pool, dev) != cudaSuccess) return;
        uint64_t keep = UINT64_MAX;   // keep freed blocks in the pool between builds
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    });
}

bool is_device_ptr(const void *p)
{
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

impact_status check_row_arrays(const impact_csr *out)
{
    if (!is_device_ptr(out->row_ptr) || !is_device_ptr(out->sink_lo) ||
        !is_device_ptr(out->sink_up) || !is_device_ptr(out->trunc))
        return fail(IMPACT_ERR_ARG, "row_ptr, sink_lo, sink_up and trunc must be device arrays");
    if (out->row_flags && !is_device_ptr(out->row_flags))
        return fail(IMPACT_ERR_ARG, "row_flags must be a device array or NULL");
    return IMPACT_OK;
}

impact_status status_result(uint32_t status)
{
    if (status & IMPACT_STATUS_TIMEOUT)
        return fail(IMPACT_ERR_TIMEOUT, "a row's look-back wait for the rows before it gave up");
    if (status & IMPACT_STATUS_INTERNAL)
        return fail(IMPACT_ERR_CUDA,
                    "internal: a row's record is damaged (the walk's step guard refused it)");
    if (status & IMPACT_STATUS_TABLE_OVERFLOW)
        return fail(IMPACT_ERR_ARG,
                    "a row's window exceeded the planner's bound (caller images wider than "
                    "128 cells in a dimension): raise the cutoff or use fewer cells");
    if (status & IMPACT_STATUS_EMIT_MISMATCH)
        return fail(IMPACT_ERR_CUDA, "internal: the emit pass disagreed with the count pass");
    if (status & IMPACT_STATUS_UNSOUND)
        return fail(IMPACT_ERR_UNSOUND, "a row check proved a row-sum invariant violated");
    return IMPACT_OK;
}

// Row outputs of build q with row-indexed arrays shifted to its first row
// (the FP64 kernels index rows from 0 within a build).
impact::RowOutputs shifted(const impact::RowOutputs &o, int64_t rb, int64_t rows_total)
{
    impact::RowOutputs s = o;
    s.row_ptr = o.row_ptr + rb;
    if (o.sink_lo) s.sink_lo = o.sink_lo + rb;
    if (o.sink_up) s.sink_up = o.sink_up + rb;
    if (o.trunc) s.trunc = o.trunc + rb;
    if (o.flags) s.flags = o.flags + rb;
    s.total_at = rows_total - rb;
    return s;
}

// FP32 walk launches of one pass over the batch's rows, in chunks of
// `chunk_rows` rows (0: one launch) in row order on `st`; `counter` is the
// pass's row counter (zero at the first launch, reset before the others).
cudaError_t walk_pass(const Batch &B, const Work &W, int mode, int warps,
                      const impact::RowOutputs &o, unsigned long long *counter,
                      int64_t chunk_rows, cudaStream_t st, bool saved = false)
{
    const int64_t step = chunk_rows > 0 ? chunk_rows : std::max<int64_t>(B.rows, 1);
    for (int64_t r0 = 0; r0 < B.rows; r0 += step) {
        cudaError_t e = r0 > 0 ? cudaMemsetAsync(counter, 0, 8, st) : cudaSuccess;
        if (e == cudaSuccess)
            e = impact::launch_walk_fp32(W.index(), r0, std::min(B.rows, r0 + step),
                                         B.rec_max, B.work_max, warps, mode, saved, o,
                                         W.lb(), B.tune.faults, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// FP64 walk launches of one pass, as walk_pass.
cudaError_t walk_pass64(const Batch &B, const Work &W, bool emit, const impact::RowOutputs &o,
                        unsigned long long *counter, int64_t chunk_rows, cudaStream_t st)
{
    const int64_t step = chunk_rows > 0 ? chunk_rows : std::max<int64_t>(B.rows, 1);
    for (int64_t r0 = 0; r0 < B.rows; r0 += step) {
        cudaError_t e = r0 > 0 ? cudaMemsetAsync(counter, 0, 8, st) : cudaSuccess;
        if (e == cudaSuccess)
            e = impact::launch_walk64(W.index(), r0, std::min(B.rows, r0 + step), B.warp64, emit, o,
                                      (double *)W.lb(), B.rows, counter, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// FP32 row records.
cudaError_t setup_pass(const Batch &B, const Work &W, cudaStream_t st)
{
    return impact::launch_setup_fp32(W.index(), B.units, B.shared32 > 0, B.shared32 < B.count(),
                                     B.item_begin.back(), W.status(), st);
}

// The builds of B into arrays of known capacity run as one walk.
bool one_pass(const Batch &B) { return B.prec == PREC_FP32_SOUND && B.tune.one_pass; }

// count pass: row_ptr (row pointers and the total), sink_lo, sink_up, trunc,
// row_flags: per-row counts, then the scan. FP64 builds whose tables are too
// large for the walk (ImpactDesc.walk64) are counted by the per-pair kernel.
impact_status run_count(const Batch &B, const Work &W, const impact_csr *out, cudaStream_t st,
                        int64_t chunk_rows, bool fresh)
{
    if (!fresh) CK(cudaMemsetAsync(W.status(), 0, 64, st));
    impact::RowOutputs o{out->row_ptr, nullptr, nullptr, nullptr, out->sink_lo, out->sink_up,
                         out->trunc, out->row_flags, W.status(), -1, B.rows};
    const impact::ScanHead scan = impact::scan_head(out->row_ptr, B.rows, W.scan(), W.total());
    if (B.prec == PREC_FP32_SOUND) {
        CK(setup_pass(B, W, st));
        CK(impact::launch_leaf_fp32(W.index(), B.leaf_begin.back(), B.leaf_smem, st));
        CK(walk_pass(B, W, WALK_COUNT, B.tune.count_warps, o, W.counter(), chunk_rows, st));
        CK(impact::launch_terms_fp32(W.index(), B.rows, W.lb(), B.tune.faults.fault_row, o, scan,
                                     st));
        CK(impact::launch_scan(out->row_ptr, B.rows, W.scan(), st, W.total(), scan.tiles > 0));
        return IMPACT_OK;
    }
    if (B.any64) {
        CK(impact::launch_items64(W.index(), B.item_begin.back(), W.status(), st));
        CK(walk_pass64(B, W, false, o, W.counter(), chunk_rows, st));
    }
    for (int q = 0; q < B.count(); ++q)
        if (!B.plans[q].desc.walk64)
            CK(impact::launch_rows(W.desc(q), B.prec, false, 0, B.plans[q].rows,
                                   shifted(o, B.row_begin[q], B.rows), st));
    if (B.any64)   // after every count: its blocks begin the scan
        CK(impact::launch_terms64(W.index(), B.rows, (const double *)W.lb(), o, scan, st));
    CK(impact::launch_scan(out->row_ptr, B.rows, W.scan(), st, W.total(),
                           B.any64 && scan.tiles > 0));
    return IMPACT_OK;
}

// emit pass at the row pointers in out->row_ptr
impact_status run_emit(const Batch &B, const Work &W, const impact_csr *out, int64_t capacity,
                       bool records_ready, cudaStream_t st, int64_t chunk_rows, bool fresh,
                       bool saved)
{
    if (!fresh) CK(cudaMemsetAsync(W.status(), 0, 64, st));
    impact::RowOutputs o{out->row_ptr, out->col, out->lo, out->up, nullptr, nullptr, nullptr,
                         nullptr, W.status(), capacity, B.rows};
    if (B.prec == PREC_FP32_SOUND) {
        if (!records_ready) {   // rebuild the records; the row outputs stay as counted
            CK(setup_pass(B, W, st));
            CK(impact::launch_leaf_fp32(W.index(), B.leaf_begin.back(), B.leaf_smem, st));
        }
        CK(walk_pass(B, W, WALK_EMIT, B.tune.emit_warps, o, W.counter() + 1, chunk_rows, st,
                     saved));
    } else {
        if (B.any64) {
            if (!records_ready)
                CK(impact::launch_items64(W.index(), B.item_begin.back(), W.status(), st));
            CK(walk_pass64(B, W, true, o, W.counter() + 1, chunk_rows, st));
        }
        for (int q = 0; q < B.count(); ++q)
            if (!B.plans[q].desc.walk64)
                CK(impact::launch_rows(W.desc(q), B.prec, true, 0, B.plans[q].rows,
                                       shifted(o, B.row_begin[q], B.rows), st));
    }
    return IMPACT_OK;
}

// the whole build into arrays of known capacity with no host round trip:
// count, scan and emit (the emit pass checks the total against the capacity
// on the device and writes nothing when it does not fit), or for FP32 with
// tuning one_pass a single walk in which each row finds its offset by the
// look-back and writes its pairs
impact_status run_fused(const Batch &B, const Work &W, const impact_csr *out, int64_t capacity,
                        cudaStream_t st, int64_t chunk_rows, bool fresh)
{
    if (!one_pass(B)) {
        impact_status s = run_count(B, W, out, st, chunk_rows, fresh);
        if (s != IMPACT_OK) return s;
        return run_emit(B, W, out, capacity, true, st, chunk_rows);
    }
    if (!fresh) CK(cudaMemsetAsync(W.status(), 0, 64, st));
    CK(setup_pass(B, W, st));
    if (B.rows > 0) CK(cudaMemsetAsync(W.lb(), 0, (size_t)B.rows * 8, st));
    else CK(cudaMemsetAsync(out->row_ptr, 0, 8, st));
    impact::RowOutputs o{out->row_ptr, out->col, out->lo, out->up, out->sink_lo, out->sink_up,
                         out->trunc, out->row_flags, W.status(), capacity, B.rows};
    CK(impact::launch_terms_fp32(W.index(), B.rows, nullptr, -1, o, impact::ScanHead(), st));
    CK(walk_pass(B, W, WALK_FUSED, B.tune.count_warps, o, W.counter(), chunk_rows, st));
    return IMPACT_OK;
}

// col/lo/up may be device memory or pinned host memory the device can
// address (the emit pass then writes the pairs straight to host memory over
// the host link); `v` is `out` with device-visible addresses.
impact_status pair_view(const impact_csr *out, impact_csr &v)
{
    v = *out;
    if (out->nnz <= 0) return IMPACT_OK;
    void **ps[3] = {(void **)&v.col, &v.lo, &v.up};
    for (void **pp : ps) {
        cudaPointerAttributes a;
        if (!*pp || cudaPointerGetAttributes(&a, *pp) != cudaSuccess) {
            cudaGetLastError();
            return fail(IMPACT_ERR_ARG, "col, lo and up must be device or pinned host arrays");
        }
        if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) continue;
        if (a.type == cudaMemoryTypeHost && a.devicePointer) {
            *pp = a.devicePointer;
            continue;
        }
        return fail(IMPACT_ERR_ARG, "col, lo and up must be device or pinned host arrays");
    }
    return IMPACT_OK;
}

// ---------------------------------------------------------------------------
// the three phases behind the entry points
// ---------------------------------------------------------------------------

// The head of the status block (Work::status), read back in one copy.
struct Outcome {
    uint32_t status = 0, abort = 0;
    int64_t nnz = 0;
};

impact_status do_count(Batch &B, impact_csr *out, cudaStream_t st)
{
    impact_status s;
    if ((s = check_row_arrays(out)) != IMPACT_OK) return s;
    configure_pool_once();
    Work W;
    if ((s = get_work(B, out, st, W)) != IMPACT_OK) return s;
    WorkHold hold{W, st};
    if (!W.owned) ws_tag(W.base, 0);
    if ((s = upload(B, W, st)) != IMPACT_OK) return s;
    if ((s = run_count(B, W, out, st, 0, true)) != IMPACT_OK) return s;
    Outcome r;
    CK(cudaMemcpyAsync(&r, W.status(), sizeof(r), cudaMemcpyDeviceToHost, st));
    if ((s = release(W, st)) != IMPACT_OK) return s;
    CK(cudaStreamSynchronize(st));
    out->rows = B.rows;
    out->nnz = r.nnz;
    s = status_result(r.status);
    if (!W.owned && (s == IMPACT_OK || s == IMPACT_ERR_UNSOUND)) ws_tag(out->workspace, B.hash);
    return s;
}

impact_status do_emit(Batch &B, impact_csr *out, cudaStream_t st)
{
    impact_status s;
    if (!is_device_ptr(out->row_ptr)) return fail(IMPACT_ERR_ARG, "row_ptr must be a device array");
    if (out->nnz < 0) return fail(IMPACT_ERR_ARG, "out->nnz (the capacity) must be >= 0");
    impact_csr view;
    if ((s = pair_view(out, view)) != IMPACT_OK) return s;
    configure_pool_once();
    bool ready = false;
    if (out->workspace) {
        if (!ws_has(out->workspace, B.hash))
            return fail(IMPACT_ERR_ARG,
                        "workspace was not filled by impact_count for these arguments");
        ready = true;
    }
    Work W;
    if ((s = get_work(B, out, st, W)) != IMPACT_OK) return s;
    WorkHold hold{W, st};
    if (!ready && (s = upload(B, W, st)) != IMPACT_OK) return s;
    if ((s = run_emit(B, W, &view, out->nnz, ready, st, 0, false, ready)) != IMPACT_OK) return s;
    uint32_t status = 0;
    CK(cudaMemcpyAsync(&status, W.status(), 4, cudaMemcpyDeviceToHost, st));
    if ((s = release(W, st)) != IMPACT_OK) return s;
    CK(cudaStreamSynchronize(st));
    out->rows = B.rows;
    if (status & IMPACT_STATUS_CAPACITY)
        return fail(IMPACT_ERR_CAPACITY, "row_ptr[rows] exceeds the capacity out->nnz");
    return status_result(status);
}

impact_status build_into(Batch &B, impact_csr *out, bool lib_owned, cudaStream_t st)
{
    impact_status s;
    const size_t vbytes = B.prec == PREC_FP32_SOUND ? 4 : 8;
    if (lib_owned) {
        CK(dev_malloc_async(&out->row_ptr, (B.rows + 1) * 8, st));
        CK(dev_malloc_async(&out->sink_lo, B.rows * 8, st));
        CK(dev_malloc_async(&out->sink_up, B.rows * 8, st));
        CK(dev_malloc_async(&out->trunc, B.rows * 8, st));
        CK(dev_malloc_async(&out->row_flags, B.rows * 4, st));
    }
    Work W;
    if (!lib_owned && one_pass(B) && !out->workspace) make_lean(B);   // it reads no leaf table
    if ((s = get_work(B, out, st, W)) != IMPACT_OK) return s;
    WorkHold hold{W, st};
    if (!W.owned) ws_tag(W.base, 0);
    if ((s = upload(B, W, st)) != IMPACT_OK) return s;
    int64_t capacity = out->nnz;
    if (lib_owned) {   // the output size is known after the count pass
        if ((s = run_count(B, W, out, st, 0, true)) != IMPACT_OK) return s;
        int64_t nnz = 0;
        CK(cudaMemcpyAsync(&nnz, W.total(), 8, cudaMemcpyDeviceToHost, st));
        CK(cudaStreamSynchronize(st));
        size_t k = (size_t)std::max<int64_t>(nnz, 1);
        CK(dev_malloc_async(&out->col, k * 4, st));
        CK(dev_malloc_async(&out->lo, k * vbytes, st));
        CK(dev_malloc_async(&out->up, k * vbytes, st));
        capacity = nnz;
        impact_csr view;
        if ((s = pair_view(out, view)) != IMPACT_OK) return s;
        if ((s = run_emit(B, W, &view, capacity, true, st)) != IMPACT_OK) return s;
    } else {   // caller capacity: no host round trip
        impact_csr view;
        if ((s = pair_view(out, view)) != IMPACT_OK) return s;
        if ((s = run_fused(B, W, &view, capacity, st, 0, true)) != IMPACT_OK) return s;
    }
    Outcome r;
    CK(cudaMemcpyAsync(&r, W.status(), sizeof(r), cudaMemcpyDeviceToHost, st));
    if ((s = release(W, st)) != IMPACT_OK) return s;
    CK(cudaStreamSynchronize(st));
    out->rows = B.rows;
    out->nnz = r.nnz;
    if (r.status & IMPACT_STATUS_CAPACITY)
        return fail(IMPACT_ERR_CAPACITY, "output capacity " + std::to_string(capacity) +
                                             " < needed pairs " + std::to_string(r.nnz));
    return status_result(r.status);
}

impact_status do_build(Batch &B, impact_csr *out, cudaStream_t st)
{
    configure_pool_once();
    const bool lib_owned = (out->col == nullptr);
    if (lib_owned) {
        void *ws = out->workspace;
        int64_t wsb = out->workspace_bytes;
        memset(out, 0, sizeof(*out));
        out->workspace = ws;
        out->workspace_bytes = wsb;
        out->owned = 1;
    } else {
        impact_status s;
        if ((s = check_row_arrays(out)) != IMPACT_OK) return s;
        if (out->nnz < 0) return fail(IMPACT_ERR_ARG, "out->nnz (the capacity) must be >= 0");
    }
    impact_status s = build_into(B, out, lib_owned, st);
    // a library-owned result that failed is released whole (an UNSOUND one is
    // complete and is kept: row_flags tells which rows)
    if (lib_owned && s != IMPACT_OK && s != IMPACT_ERR_UNSOUND) {
        std::string msg = g_last_error;
        free_owned(out, st);
        cudaStreamSynchronize(st);
        fail(s, msg);
    }
    return s;
}

impact_request single(const impact_system *sys, const impact_grid *grid,
                      const impact_inputs *inputs, const double *sigma, double cutoff)
{
    impact_request r;
    r.sys = sys;
    r.grid = grid;
    r.inputs = inputs;
    r.sigma = sigma;
    r.cutoff = cutoff;
    return r;
}

impact_status check_request_ptrs(const impact_request *reqs, int count)
{
    if (!reqs) return fail(IMPACT_ERR_ARG, "null request array");
    for (int q = 0; q < count; ++q)
        if (!reqs[q].sys || !reqs[q].grid || !reqs[q].inputs || !reqs[q].sigma)
            return fail(IMPACT_ERR_ARG, "request " + std::to_string(q) + ": null argument");
    return IMPACT_OK;
}

static_assert(IMPACT_REGION_BOXES == IMPACT_REGION_MAX_BOXES, "region box limits differ");

// Region boxes -> blocks of whole cells: in every dimension the cells whose
// centre (midpoint of the cell's edges, edges as the planner makes them)
// lies in the closed box. Boxes with no such cell are dropped; targets stay
// first. `disjoint`: refuse boxes that share a cell.
impact_status snap_regions(const impact_grid *grid, const impact_regions *reg, bool disjoint,
                           RegionBoxes &B)
{
    if (!grid || !grid->lo || !grid->hi || !grid->cells) return fail(IMPACT_ERR_ARG, "null grid");
    const int n = grid->n;
    if (n < 1 || n > IMPACT_MAX_DIM) return fail(IMPACT_ERR_ARG, "grid.n must be in [1, 8]");
    int64_t total = 1;
    for (int d = 0; d < n; ++d) {
        if (grid->cells[d] < 1) return fail(IMPACT_ERR_ARG, "cells must be >= 1");
        if (!(grid->lo[d] < grid->hi[d]) || !isfinite(grid->lo[d]) || !isfinite(grid->hi[d]))
            return fail(IMPACT_ERR_ARG, "grid needs finite lo < hi");
        total *= grid->cells[d];
        if (total >= ((int64_t)1 << 31)) return fail(IMPACT_ERR_ARG, "more than 2^31-1 cells");
    }
    if (!reg) return fail(IMPACT_ERR_ARG, "null regions");
    const int nt = reg->n_target, na = reg->n_avoid;
    if (nt < 0 || na < 0 || nt + na > IMPACT_REGION_MAX_BOXES)
        return fail(IMPACT_ERR_ARG, "region boxes: 0 <= n_target + n_avoid <= 16");
    if ((nt > 0 && (!reg->target_lo || !reg->target_hi)) ||
        (na > 0 && (!reg->avoid_lo || !reg->avoid_hi)))
        return fail(IMPACT_ERR_ARG, "null region box corners");
    memset(&B, 0, sizeof(B));
    B.n = n;
    for (int d = 0; d < n; ++d) B.cells[d] = grid->cells[d];
    for (int k = 0; k < nt + na; ++k) {
        const bool avoid = k >= nt;
        const double *lo = avoid ? reg->avoid_lo + (size_t)(k - nt) * n : reg->target_lo + (size_t)k * n;
        const double *hi = avoid ? reg->avoid_hi + (size_t)(k - nt) * n : reg->target_hi + (size_t)k * n;
        bool empty = false;
        for (int d = 0; d < n; ++d) {
            if (!isfinite(lo[d]) || !isfinite(hi[d]) || lo[d] > hi[d])
                return fail(IMPACT_ERR_ARG, "region boxes need finite lo <= hi");
            const int N = grid->cells[d];
            const double h = (grid->hi[d] - grid->lo[d]) / (double)N;
            auto edge = [&](int i) { return i >= N ? grid->hi[d] : grid->lo[d] + (double)i * h; };
            int f = -1, l = -2;
            for (int i = 0; i < N; ++i) {
                const double c = 0.5 * (edge(i) + edge(i + 1));
                if (c >= lo[d] && c <= hi[d]) {
                    if (f < 0) f = i;
                    l = i;
                }
            }
            if (f < 0) empty = true;
            B.first[B.count][d] = f;
            B.last[B.count][d] = l;
        }
        if (empty) continue;
        if (!avoid) ++B.n_target;
        ++B.count;
    }
    if (disjoint)
        for (int a = 0; a < B.count; ++a)
            for (int b = 0; b < a; ++b) {
                bool meet = true;
                for (int d = 0; d < n; ++d)
                    meet = meet && std::max(B.first[a][d], B.first[b][d]) <=
                                       std::min(B.last[a][d], B.last[b][d]);
                if (meet) return fail(IMPACT_ERR_ARG, "region boxes share cells");
            }
    return IMPACT_OK;
}

}  // namespace impact

using namespace impact;

// A captured pipeline: count, scan and emit of one batch into fixed caller
// buffers, replayed by impact_graph_launch.
struct impact_graph {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    impact::Outcome *h_result = nullptr;   // pinned
    unsigned char *own_ws = nullptr;
    int64_t rows = 0, capacity = 0;
};

extern "C" {

impact_status impact_plan(const impact_system *sys, const impact_grid *grid,
                          const impact_inputs *inputs, const double *sigma, double cutoff,
                          impact_precision precision, int64_t *rows, int64_t *nnz_upper_bound,
                          int64_t *bytes_upper_bound)
{
    impact_request r = single(sys, grid, inputs, sigma, cutoff);
    Batch B;
    impact_status s = make_batch(&r, 1, precision, nullptr, B);
    if (s != IMPACT_OK) return s;
    if (rows) *rows = B.rows;
    if (nnz_upper_bound) *nnz_upper_bound = B.nnz_bound;
    if (bytes_upper_bound) {
        int64_t per_pair = precision == IMPACT_FP32_SOUND ? 12 : 20;
        *bytes_upper_bound = B.nnz_bound * per_pair + (B.rows + 1) * 8 + B.rows * (3 * 8 + 4) +
                             (int64_t)batch_layout(B).total;
    }
    return IMPACT_OK;
}

impact_status impact_workspace_bytes(const impact_system *sys, const impact_grid *grid,
                                     const impact_inputs *inputs, const double *sigma,
                                     double cutoff, impact_precision precision, int64_t *bytes)
{
    impact_request r = single(sys, grid, inputs, sigma, cutoff);
    Batch B;
    impact_status s = make_batch(&r, 1, precision, nullptr, B);
    if (s != IMPACT_OK) return s;
    if (bytes) *bytes = (int64_t)batch_layout(B).total;
    return IMPACT_OK;
}

impact_status impact_count(const impact_system *sys, const impact_grid *grid,
                           const impact_inputs *inputs, const double *sigma, double cutoff,
                           impact_precision precision, impact_csr *out, void *stream)
{
    if (!out) return fail(IMPACT_ERR_ARG, "null output");
    impact_request r = single(sys, grid, inputs, sigma, cutoff);
    Batch B;
    impact_status s = make_batch(&r, 1, precision, nullptr, B);
    if (s != IMPACT_OK) return s;
    return do_count(B, out, (cudaStream_t)stream);
}

impact_status impact_emit(const impact_system *sys, const impact_grid *grid,
                          const impact_inputs *inputs, const double *sigma, double cutoff,
                          impact_precision precision, impact_csr *out, void *stream)
{
    if (!out) return fail(IMPACT_ERR_ARG, "null output");
    impact_request r = single(sys, grid, inputs, sigma, cutoff);
    Batch B;
    impact_status s = make_batch(&r, 1, precision, nullptr, B);
    if (s != IMPACT_OK) return s;
    return do_emit(B, out, (cudaStream_t)stream);
}

impact_status impact_build(const impact_system *sys, const impact_grid *grid,
                           const impact_inputs *inputs, const double *sigma, double cutoff,
                           impact_precision precision, impact_csr *out, void *stream)
{
    if (!out) return fail(IMPACT_ERR_ARG, "null output");
    impact_request r = single(sys, grid, inputs, sigma, cutoff);
    Batch B;
    impact_status s = make_batch(&r, 1, precision, nullptr, B);
    if (s != IMPACT_OK) return s;
    return do_build(B, out, (cudaStream_t)stream);
}

impact_status impact_batch_plan(const impact_request *reqs, int count, impact_precision precision,
                                const impact_tuning *tuning, int64_t *row_offsets,
                                int64_t *nnz_upper_bound, int64_t *workspace_bytes,
                                int64_t *upload_bytes)
{
    impact_status s = check_request_ptrs(reqs, count);
    if (s != IMPACT_OK) return s;
    Batch B;
    if ((s = make_batch(reqs, count, precision, tuning, B)) != IMPACT_OK) return s;
    if (row_offsets) memcpy(row_offsets, B.row_begin.data(), (size_t)(count + 1) * 8);
    if (nnz_upper_bound) *nnz_upper_bound = B.nnz_bound;
    if (workspace_bytes || upload_bytes) {
        const BatchLayout L = batch_layout(B);
        if (workspace_bytes) *workspace_bytes = (int64_t)L.total;
        if (upload_bytes) *upload_bytes = (int64_t)L.upload_end;
    }
    return IMPACT_OK;
}

impact_status impact_batch_count(const impact_request *reqs, int count,
                                 impact_precision precision, const impact_tuning *tuning,
                                 impact_csr *out, void *stream)
{
    if (!out) return fail(IMPACT_ERR_ARG, "null output");
    impact_status s = check_request_ptrs(reqs, count);
    if (s != IMPACT_OK) return s;
    Batch B;
    if ((s = make_batch(reqs, count, precision, tuning, B)) != IMPACT_OK) return s;
    return do_count(B, out, (cudaStream_t)stream);
}

impact_status impact_batch_emit(const impact_request *reqs, int count,
                                impact_precision precision, const impact_tuning *tuning,
                                impact_csr *out, void *stream)
{
    if (!out) return fail(IMPACT_ERR_ARG, "null output");
    impact_status s = check_request_ptrs(reqs, count);
    if (s != IMPACT_OK) return s;
    Batch B;
    if ((s = make_batch(reqs, count, precision, tuning, B)) != IMPACT_OK) return s;
    return do_emit(B, out, (cudaStream_t)stream);
}

impact_status impact_batch_build(const impact_request *reqs, int count,
                                 impact_precision precision, const impact_tuning *tuning,
                                 impact_csr *out, void *stream)
{
    if (!out) return fail(IMPACT_ERR_ARG, "null output");
    impact_status s = check_request_ptrs(reqs, count);
    if (s != IMPACT_OK) return s;
    Batch B;
    if ((s = make_batch(reqs, count, precision, tuning, B)) != IMPACT_OK) return s;
    return do_build(B, out, (cudaStream_t)stream);
}

impact_status impact_graph_create(const impact_request *reqs, int count,
                                  impact_precision precision, const impact_tuning *tuning,
                                  const impact_csr *out, void *stream, impact_graph **graph)
{
    if (!out || !graph) return fail(IMPACT_ERR_ARG, "null output or graph handle");
    *graph = nullptr;
    impact_status s = check_request_ptrs(reqs, count);
    if (s != IMPACT_OK) return s;
    Batch B;
    if ((s = make_batch(reqs, count, precision, tuning, B)) != IMPACT_OK) return s;
    if ((s = check_row_arrays(out)) != IMPACT_OK) return s;
    if (!out->col) return fail(IMPACT_ERR_ARG, "a graph writes into caller-owned col/lo/up");
    if (out->nnz < 0) return fail(IMPACT_ERR_ARG, "out->nnz (the capacity) must be >= 0");
    impact_csr view;
    if ((s = pair_view(out, view)) != IMPACT_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    impact_graph *g = new impact_graph();
    g->rows = B.rows;
    g->capacity = out->nnz;
    Work W;
    if (one_pass(B) && !out->workspace) make_lean(B);   // it reads no leaf table
    W.L = batch_layout(B);
    auto cleanup = [&](impact_status r) {
        if (g->exec) cudaGraphExecDestroy(g->exec);
        if (g->graph) cudaGraphDestroy(g->graph);
        host_free(g->h_result);
        dev_free(g->own_ws);
        delete g;
        return r;
    };
    if (out->workspace) {
        if (out->workspace_bytes < (int64_t)W.L.total || ((uintptr_t)out->workspace & 255))
            return cleanup(fail(IMPACT_ERR_ARG, "workspace too small or not 256-byte aligned"));
        W.base = (unsigned char *)out->workspace;
        ws_tag(W.base, 0);
    } else {
        cudaError_t e = dev_malloc(&g->own_ws, W.L.total);
        if (e == cudaErrorMemoryAllocation && make_lean(B)) {
            W.L = batch_layout(B);
            e = dev_malloc(&g->own_ws, W.L.total);
        }
        if (e != cudaSuccess) return cleanup(fail(IMPACT_ERR_OOM, cudaGetErrorString(e)));
        W.base = g->own_ws;
    }
    if (host_malloc(&g->h_result, sizeof(Outcome)) != cudaSuccess)
        return cleanup(fail(IMPACT_ERR_OOM, "pinned result word"));
    if ((s = upload(B, W, st)) != IMPACT_OK) return cleanup(s);
    if (cudaStreamSynchronize(st) != cudaSuccess)
        return cleanup(fail(IMPACT_ERR_CUDA, "upload before capture failed"));
    // capture on a private stream: the caller's may be the legacy default one
    cudaStream_t cs = nullptr;
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess)
        return cleanup(fail(IMPACT_ERR_CUDA, "capture stream"));
    impact_csr o = view;
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeRelaxed);
    if (e == cudaSuccess) {
        s = run_fused(B, W, &o, g->capacity, cs);
        if (s == IMPACT_OK) {
            cudaMemcpyAsync(g->h_result, W.status(), sizeof(Outcome), cudaMemcpyDeviceToHost, cs);
        }
        cudaError_t e2 = cudaStreamEndCapture(cs, &g->graph);
        if (s == IMPACT_OK && e2 != cudaSuccess) s = fail(IMPACT_ERR_CUDA, cudaGetErrorString(e2));
    } else {
        s = fail(IMPACT_ERR_CUDA, cudaGetErrorString(e));
    }
    cudaStreamDestroy(cs);
    if (s != IMPACT_OK) return cleanup(s);
    e = cudaGraphInstantiate(&g->exec, g->graph, 0);
    if (e != cudaSuccess) return cleanup(fail(IMPACT_ERR_CUDA, cudaGetErrorString(e)));
    *graph = g;
    return IMPACT_OK;
}

impact_status impact_graph_launch(impact_graph *graph, void *stream)
{
    if (!graph || !graph->exec) return fail(IMPACT_ERR_ARG, "null graph");
    graph->h_result->nnz = -1;
    graph->h_result->status = 0;
    CK(cudaGraphLaunch(graph->exec, (cudaStream_t)stream));
    return IMPACT_OK;
}

impact_status impact_graph_result(impact_graph *graph, int64_t *nnz)
{
    if (!graph) return fail(IMPACT_ERR_ARG, "null graph");
    const int64_t got = graph->h_result->nnz;
    const uint32_t status = graph->h_result->status;
    if (nnz) *nnz = got;
    if (got < 0) return fail(IMPACT_ERR_ARG, "no finished launch: synchronize the stream first");
    if (status & IMPACT_STATUS_CAPACITY)
        return fail(IMPACT_ERR_CAPACITY, "output capacity " + std::to_string(graph->capacity) +
                                             " < needed pairs " + std::to_string(got));
    return status_result(status);
}

impact_status impact_graph_destroy(impact_graph *graph)
{
    if (!graph) return IMPACT_OK;
    if (graph->exec) cudaGraphExecDestroy(graph->exec);
    if (graph->graph) cudaGraphDestroy(graph->graph);
    host_free(graph->h_result);
    dev_free(graph->own_ws);
    delete graph;
    return IMPACT_OK;
}

impact_status impact_batch_tune(const impact_request *reqs, int count,
                                impact_precision precision, impact_csr *out, int reps,
                                void *stream, impact_tuning *best, double *best_ms)
{
    if (!out || !best) return fail(IMPACT_ERR_ARG, "null output or result");
    if (precision != IMPACT_FP32_SOUND)
        return fail(IMPACT_ERR_ARG, "the autotuner tunes the FP32-sound walk");
    impact_status s = check_request_ptrs(reqs, count);
    if (s != IMPACT_OK) return s;
    if ((s = check_row_arrays(out)) != IMPACT_OK) return s;
    impact_csr view;
    if ((s = pair_view(out, view)) != IMPACT_OK) return s;
    out = &view;
    reps = std::max(1, std::min(reps, 50));
    cudaStream_t st = (cudaStream_t)stream;
    configure_pool_once();
    Batch B0;
    if ((s = make_batch(reqs, count, precision, nullptr, B0)) != IMPACT_OK) return s;
    Work W;
    impact_csr wout = *out;
    wout.workspace = nullptr;   // the tuner keeps its own scratch
    if ((s = get_work(B0, &wout, st, W)) != IMPACT_OK) return s;
    WorkHold hold{W, st};
    if ((s = upload(B0, W, st)) != IMPACT_OK) return s;
    if ((s = run_count(B0, W, out, st)) != IMPACT_OK) return s;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    // pass 0: count, 1: emit
    auto timed = [&](int warps, int pass, double &ms) -> impact_status {
        Batch B = B0;
        B.tune.count_warps = B.tune.emit_warps = warps;
        ms = 1e30;
        for (int i = 0; i < reps; ++i) {
            CK(cudaEventRecord(e0, st));
            impact_status r = pass == 0 ? run_count(B, W, out, st)
                                        : run_emit(B, W, out, out->nnz, true, st, 0, false);
            if (r != IMPACT_OK) return r;
            CK(cudaEventRecord(e1, st));
            CK(cudaEventSynchronize(e1));
            float f = 0.0f;
            CK(cudaEventElapsedTime(&f, e0, e1));
            ms = std::min(ms, (double)f);
        }
        uint32_t status = 0;
        CK(cudaMemcpy(&status, W.status(), 4, cudaMemcpyDeviceToHost));
        if (status & ~IMPACT_STATUS_UNSOUND) ms = 1e30;   // a shape that cannot run this batch
        return IMPACT_OK;
    };
    const bool can_emit = out->col != nullptr;
    const int warps[4] = {2, 4, 6, 8};
    impact_tuning tb;
    memset(&tb, 0, sizeof(tb));
    double best_a = 1e30, best_b = 1e30;
    // the count shape, then (with output arrays) the emit shape
    for (int w : warps) {
        double ms;
        if ((s = timed(w, 0, ms)) != IMPACT_OK) break;
        if (ms < best_a) {
            best_a = ms;
            tb.count_warps = w;
        }
    }
    if (s == IMPACT_OK && can_emit)
        for (int w : warps) {
            double ms;
            if ((s = timed(w, 1, ms)) != IMPACT_OK) break;
            if (ms < best_b) {
                best_b = ms;
                tb.emit_warps = w;
            }
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    impact_status r2 = release(W, st);
    if (s != IMPACT_OK) return s;
    if (r2 != IMPACT_OK) return r2;
    if (best_a >= 1e30) return fail(IMPACT_ERR_ARG, "no launch shape ran this batch");
    if (tb.emit_warps == 0) tb.emit_warps = IMPACT_TREE_WARPS;
    *best = tb;
    if (best_ms) *best_ms = best_a + (can_emit && best_b < 1e30 ? best_b : 0.0);
    return IMPACT_OK;
}

impact_status impact_free(impact_csr *out)
{
    if (!out) return fail(IMPACT_ERR_ARG, "null output");
    if (!out->owned) return IMPACT_OK;
    void *ptrs[] = {out->row_ptr, out->col, out->lo, out->up, out->sink_lo,
                    out->sink_up, out->trunc, out->row_flags};
    for (void *p : ptrs)
        if (p) CK(dev_free(p));
    void *ws = out->workspace;
    int64_t wsb = out->workspace_bytes;
    memset(out, 0, sizeof(*out));
    out->workspace = ws;
    out->workspace_bytes = wsb;
    return IMPACT_OK;
}

const char *impact_last_error(void) { return g_last_error.c_str(); }

impact_status impact_label_cells(const impact_grid *grid, const impact_regions *regions,
                                 uint8_t *labels, void *stream)
{
    RegionBoxes B;
    impact_status s = snap_regions(grid, regions, false, B);
    if (s != IMPACT_OK) return s;
    if (!is_device_ptr(labels)) return fail(IMPACT_ERR_ARG, "labels must be a device array");
    int64_t total = 1;
    for (int d = 0; d < grid->n; ++d) total *= grid->cells[d];
    cudaError_t e = launch_labels(B, total, labels, (cudaStream_t)stream);
    if (e != cudaSuccess) return fail(IMPACT_ERR_CUDA, cudaGetErrorString(e));
    return IMPACT_OK;
}

impact_status impact_region_vectors(const impact_system *sys, const impact_grid *grid,
                                    const impact_inputs *inputs, const double *sigma,
                                    const impact_regions *regions, impact_region_mode mode,
                                    impact_precision precision, double *r_lo, double *r_up,
                                    double *a_lo, double *a_up, void *stream)
{
    if (mode != IMPACT_REGION_BOX && mode != IMPACT_REGION_CELL_SUM)
        return fail(IMPACT_ERR_ARG, "unknown region mode");
    if (precision != IMPACT_FP32_SOUND && precision != IMPACT_FP64_PLAIN)
        return fail(IMPACT_ERR_ARG, "unknown precision");
    if (!sys || !grid || !inputs || !sigma) return fail(IMPACT_ERR_ARG, "null argument");
    RegionBoxes B;
    impact_status s = snap_regions(grid, regions, true, B);
    if (s != IMPACT_OK) return s;
    if (!is_device_ptr(r_lo) || !is_device_ptr(r_up) || !is_device_ptr(a_lo) ||
        !is_device_ptr(a_up))
        return fail(IMPACT_ERR_ARG, "the region vectors must be device arrays");
    configure_pool_once();
    cudaStream_t st = (cudaStream_t)stream;
    // the FP64 tables of the build (images in both roundings); the cutoff
    // does not enter the vectors, and one near 1 keeps the planner's windows
    // small
    impact_request req = single(sys, grid, inputs, sigma, 0.999);
    Batch batch;
    s = make_batch(&req, 1, IMPACT_FP64_PLAIN, nullptr, batch);
    if (s != IMPACT_OK) return s;
    batch.walks = false;
    batch.extra = region_scratch(batch.plans[0].desc, B);
    Work W;
    s = get_work(batch, nullptr, st, W);
    if (s == IMPACT_ERR_OOM && batch.extra >= kSpareMin) {
        batch.extra = 0;
        s = get_work(batch, nullptr, st, W);
    }
    if (s != IMPACT_OK) return s;
    WorkHold hold{W, st};
    s = upload(batch, W, st);
    if (s == IMPACT_OK) {
        cudaError_t e = launch_regions(batch.plans[0].desc, W.desc(0), batch.rows, B,
                                       mode == IMPACT_REGION_CELL_SUM,
                                       precision == IMPACT_FP32_SOUND,
                                       batch.extra > 0 ? W.base + W.L.extra : nullptr, r_lo, r_up,
                                       a_lo, a_up, st);
        if (e != cudaSuccess) s = fail(IMPACT_ERR_CUDA, cudaGetErrorString(e));
    }
    impact_status r = release(W, st);
    return s != IMPACT_OK ? s : r;
}

int impact_version(void) { return 301; }

}  // extern "C"
