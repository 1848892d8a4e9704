// pipeline.h -- a batch of builds, its device workspace and the count /
// emit pipeline (api.cu), shared with the serving runtime (server.cu);
// internal.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/impact.h"
#include "impact_desc.h"
#include "kernels.h"
#include "plan.h"

namespace impact {

struct Batch {
    std::vector<Plan> plans;
    std::vector<const double *> images;   // per build: device images (IMAGES kind)
    std::vector<int64_t> row_begin;       // [count + 1] first global row of each build
    std::vector<int64_t> unit_begin;      // [count + 1] first setup unit (32/n rows)
    int64_t rows = 0, units = 0, nnz_bound = 0;
    int prec = 0;
    int rec_max = 0;                      // FP32 walk: largest record of the batch
    int work_max[3] = {0, 0, 0};          // FP32 walk: largest work space per mode
    bool walks = true;                    // false: only the tables are used (no walk scratch)
    int64_t extra = 0;                    // bytes of the call's own scratch
    int any64 = 0, warp64 = 0;            // FP64 walk: builds on it, largest warp memory
    int shared32 = 0, leaf_smem = 0;      // FP32: builds with shared windows, leaf kernel memory
    std::vector<int64_t> item_begin;      // [count * IMPACT_MAX_DIM + 1] first item unit
    std::vector<int64_t> leaf_begin;      // [count + 1] first leaf table
    Tuning tune;
    uint64_t hash = 0;
    int count() const { return (int)plans.size(); }
};

impact_status make_batch(const impact_request *reqs, int count, impact_precision precision,
                         const impact_tuning *tuning, Batch &B);

// Plans the builds `only` (or all, < 0) again without the tables that only save
// time, FP64 items and FP32 leaf tables: the per-pair kernel and per-row tables
// take their place, as at sizes beyond them (the same pairs; the FP64 truncated
// mass is summed in another order). False: too little to give up.
bool make_lean(Batch &B, int only = -1);
// Scratch that a call can do without and whose lack is worth a second try.
constexpr int64_t kSpareMin = (int64_t)16 << 20;

// Offsets (bytes, 256-aligned) of everything in the device workspace.
struct BatchLayout {
    size_t index = 0, row_begin = 0, unit_begin = 0, descs = 0, recs = 0, item_begin = 0;
    size_t items = 0, leafs = 0, termps = 0, leaf_begin = 0;
    std::vector<size_t> tables;            // per build: its descriptor and tables
    std::vector<impact::TableLayout> tl;
    size_t upload_end = 0;                 // [0, upload_end) is copied from the host
    size_t status = 0, scan = 0;
    size_t lb = 0;                         // per row: 16 bytes (FP32 look-back word, or the
                                           // count's sums), 24 (FP64 sums)
    std::vector<size_t> rec;               // per build: FP32 per-row records
    std::vector<size_t> item, leaf;        // per build: item tables, FP32 leaf tables
    std::vector<size_t> term;              // per build: FP32 (row, dimension) numbers
    size_t extra = 0;                      // the call's own scratch
    size_t total = 0;
};

BatchLayout batch_layout(const Batch &B);

// The device workspace of one call.
struct Work {
    unsigned char *base = nullptr;
    BatchLayout L;
    bool owned = false;
    const BatchIndex *index() const { return (const BatchIndex *)(base + L.index); }
    // 64 bytes: the status word and the look-back abort flag, the pair total,
    // the row counters of the count and the emit walk
    uint32_t *status() const { return (uint32_t *)(base + L.status); }
    int64_t *total() const { return (int64_t *)(base + L.status) + 1; }
    unsigned long long *counter() const { return (unsigned long long *)(base + L.status) + 2; }
    int64_t *scan() const { return (int64_t *)(base + L.scan); }
    unsigned long long *lb() const { return (unsigned long long *)(base + L.lb); }
    const ImpactDesc *desc(int q) const
    {
        return (const ImpactDesc *)(base + L.tables[q] + L.tl[q].desc);
    }
};

// Copies the batch index, the descriptors, the tables and a zeroed status block
// into W (stream-ordered).
impact_status upload(const Batch &B, Work &W, cudaStream_t st);
// The passes below launch the walks over all rows at once, or in chunks of
// `chunk_rows` rows one after another on `st` (so that work on other streams can
// take SMs between chunks); the per-pair FP64 kernel ignores chunk_rows.
// count pass into out's row arrays (row pointers included). `fresh`: W's status
// block is as an upload left it (zeroed).
impact_status run_count(const Batch &B, const Work &W, const impact_csr *out, cudaStream_t st,
                        int64_t chunk_rows = 0, bool fresh = false);
// emit pass into out's pair arrays at the row pointers of a count pass
// (`records_ready`: W holds the records or items of that count pass; `saved`:
// the caller has held W since; `fresh`: W's status block is as a count left it,
// or zeroed).
impact_status run_emit(const Batch &B, const Work &W, const impact_csr *out, int64_t capacity,
                       bool records_ready, cudaStream_t st, int64_t chunk_rows = 0,
                       bool fresh = true, bool saved = false);
// The whole build into arrays of known capacity (`fresh` as in run_count).
impact_status run_fused(const Batch &B, const Work &W, const impact_csr *out, int64_t capacity,
                        cudaStream_t st, int64_t chunk_rows = 0, bool fresh = false);
// Maps the device status word of a finished pipeline to a status code.
impact_status status_result(uint32_t status);
void configure_pool_once();

}  // namespace impact
