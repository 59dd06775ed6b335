// Internal declarations shared by the translation units of libws.so.
// Nothing here is part of the public ABI (see include/ws.h).
#pragma once
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include <vector>

#include "ws.h"

// A named range around an entry point for timeline tools (NVTX; costs a few nanoseconds when no tool
// is attached).  Covers the host side of the call: argument checks and launches.
struct WsRange {
    explicit WsRange(const char* name) { nvtxRangePushA(name); }
    ~WsRange() { nvtxRangePop(); }
    WsRange(const WsRange&) = delete;
    WsRange& operator=(const WsRange&) = delete;
};

// One work tile: a run of at most `tile_elems` consecutive shard positions that
// lies inside one tensor's piece.  A tile carries everything a kernel needs to
// address and mask its elements, so the kernels never search the segment table.
//   shard position of element e of the tile : pos + e
//   index of that element in tensor `seg`    : r*piece + poff + e      (shard r)
//   it exists in the tensor iff              : e < vt - r*piece
// Per-tensor layout: one tile list serves every shard r.  Concatenated layout: every shard
// has its own tiles (`shard` says which), piece is 0 and poff / vt are absolute.
struct __align__(16) WsTile {
    long long pos;    // start inside a shard, multiple of 8
    long long vt;     // numel - poff: valid elements from the tile start in shard 0
    long long piece;  // p_t
    long long poff;   // pos - off_t: start inside the piece
    int len;          // elements in the tile, multiple of 8, <= tile_elems
    int seg;          // tensor index t
    int shard;        // concatenated layout only: the shard this tile lies in
    int pad1;
};
static_assert(sizeof(WsTile) == 48, "WsTile is read as three 16-byte words");

// Per tensor: which tiles of a shard belong to it (contiguous range).
struct WsSegTiles {
    int tile_begin;
    int tile_count;
};

// Adafactor's view of a tensor: foff = start of its factored state (floats); nrow row
// accumulators (0 for an unfactored tensor) followed by ncol column accumulators (the full
// second moment for an unfactored tensor, which is handled as a single row).
struct WsSegAf {
    long long foff;
    long long nrow;
    long long ncol;
    long long numel;
    // the workspace arrays (this step's sums, the 1/sqrt factors) use a padded layout so that a
    // thread's run of columns can be moved as one vector: row part and column part each start on
    // a multiple of 8 floats
    long long irow;
    long long icol;
};

// The finalize steps walk the factored state in chunks of at most 1024 entries (one CTA each).
struct WsAfChunk {
    long long begin;   // first entry inside tensor seg's state (0 .. nrow + ncol)
    int count;
    int seg;
};

// One-launch schedule of the norm-based optimizers (LAMB, LARS): the update of all shards as ONE
// kernel.  A work item is one or several consecutive whole tiles of a tensor in one shard; every item
// appears twice in the schedule, once for phase 1 (reduce, moments, partial norm sums of every tile)
// and once for phase 2 (apply the step with the tensor's ratio).
constexpr int kWsItemElems = 8192;    // an item of several tiles has at most this many elements
constexpr int kWsItemTiles = 8;       // ... and tiles
struct __align__(16) WsItem {
    unsigned long long pos_shard;   // (start inside the shard, multiple of 8) << 16 | shard
    long long toff;       // element index of the first element inside tensor `seg`
    int seg;              // tensor index
    int nvalid;           // elements of the item that exist in the tensor (the rest is padding)
    int len;              // elements, multiple of 8
    int tile;             // its first tile (per-tensor layout: of the shard's; concatenated: of all)
};
static_assert(sizeof(WsItem) == 32, "WsItem is read as two 16-byte words");
// Items are numbered tensor by tensor (then shard by shard): a tensor's items are one contiguous range.
struct __align__(16) WsItemSeg {
    int first;
    int count;
    int tile_begin;       // its tiles, as in WsSegTiles
    int tile_count;
};

// Adafactor's all-shard update as one kernel (ws_af_onelaunch.cu).  A work item is a block of a tensor's
// rows x cols matrix: 256 threads as rp rows of tpr threads, a thread owning 8 columns (4 where the row
// length is no multiple of 8) and walking down the rows, so that its column sums live in registers for the
// whole block.
enum { WS_AF_VEC8 = 0, WS_AF_VEC4 = 1, WS_AF_SCALAR = 2, WS_AF_FULL = 3, WS_AF_NARROW = 4 };
__host__ __device__ constexpr int ws_af_width(int mode) { return mode == WS_AF_VEC8 ? 8 : 4; }   // columns per thread
// Rows that 4 does not divide: a thread's 4 columns are scalar accesses, but one vector in the kept sums, whose places
// beyond the row stay empty.  Where those would be more than an eighth of the row (a row of one column would take four
// times its size) the sums are kept element by element too: WS_AF_NARROW.
__host__ __device__ constexpr bool ws_af_scalar(int mode) { return mode == WS_AF_SCALAR || mode == WS_AF_NARROW; }
// Floats that a row of a block takes in the kept sums.
__host__ __device__ constexpr int ws_af_kept_row(int mode, int nc, int tpr) {
    return mode == WS_AF_NARROW ? nc : tpr * ws_af_width(mode);
}
constexpr int kWsAfChunk = 1024;      // state entries per moments entry
// One record per schedule entry, in execution order, so that a CTA reads its work with one access.
struct __align__(16) WsAfItem {
    int seg;               // tensor index
    int row0, col0;        // first row and column of the block
    unsigned goff32;       // where the block's summed gradients are kept, in units of 32 floats
    unsigned short nr;     // rows of the block
    unsigned short nc;     // columns of the block, <= 8 tpr (4 tpr)
    unsigned short tpr;    // threads per row
    unsigned short rp;     // rows in parallel
    unsigned item;         // index of the block (partial sums)
    int phase;             // 0: sums, 1: moments (row0, col0: first state entry, low and high half; goff32: entries), 2: U^2, 3: apply
};
static_assert(sizeof(WsAfItem) == 32, "WsAfItem is read as two 16-byte words");
struct __align__(16) WsAfTensor {
    long long numel, ncol, nrow;      // WS_AF_FULL: ncol is the length of the virtual rows the items walk
    long long foff, irow, icol;       // factored state and its padded workspace layout, as in WsSegAf
    long long piece, off;             // packed position of element e: (e / piece) S + off + e % piece
    long long pad_end;                // concatenated layout: its pads are elements [numel, pad_end)
    int item_first, item_count, chunk_count, mode;
    long long rfac;                   // start of its 64-bit row factors
};
static_assert(sizeof(WsAfTensor) == 96, "WsAfTensor is read as six 16-byte words");

struct ws_plan {
    int T = 0, R = 0, A = 0, K = 0;
    int layout = 0;                           // ws_layout
    long long S = 0, N = 0;
    long long ntiles = 0;                     // per-tensor layout: tiles per shard; concatenated: all tiles
    int longest = 0;                          // elements of the longest tile (at most K)
    std::vector<long long> shard_tile_begin;  // concatenated layout: [R+1] first tile of every shard
    std::vector<ws_segment> segs;
    std::vector<WsTile> tiles;
    std::vector<WsSegTiles> segtiles;
    // tensor arena: tensors back to back, each start rounded up to 8 elements
    std::vector<long long> arena_off;
    long long arena_elems = 0;
    // images of small uploads; they live as long as the plan, since a captured copy reads its source at every replay
    std::vector<char> table_image, sched_image;
    // device copies (caller-owned memory, set by ws_plan_upload)
    int sms = 148;                            // multiprocessors of the device of the upload
    const WsTile* d_tiles = nullptr;
    const WsSegTiles* d_segtiles = nullptr;
    std::vector<WsSegAf> segaf;
    std::vector<WsAfChunk> afchunks;
    long long F = 0;                          // total factored-state floats
    long long Fi = 0;                         // floats of the padded workspace layout
    const WsSegAf* d_segaf = nullptr;
    const WsAfChunk* d_afchunks = nullptr;
    // one-launch schedule: counted at creation, built and uploaded by ws_plan_upload_schedule
    long long n_items = 0;                    // work items (0: the plan has no one-launch schedule)
    std::vector<WsItem> items;
    std::vector<WsItemSeg> itemsegs;          // [T]
    std::vector<unsigned> sched;              // [2 n_items]: item index * 2 + phase, in execution order
    // the same for Adafactor (0 items: the plan has none)
    long long n_afitems = 0, n_afsched = 0, af_ghat = 0, af_rows = 0;   // items, schedule entries, floats of kept gradient sums, rows
    long long af_scalar = 0;                  // elements in rows that 4 does not divide
    std::vector<WsAfTensor> aftensors;
    std::vector<WsAfItem> afsched;
    const WsAfTensor* d_aftensors = nullptr;
    const WsAfItem* d_afsched = nullptr;
    const WsItem* d_items = nullptr;
    const WsItemSeg* d_itemsegs = nullptr;
    const unsigned* d_sched = nullptr;
};

// Optimizer constants narrowed to fp32 for the kernels.
struct WsConsts {
    float lr, beta1, omb1, beta2, omb2, eps, wd, mu, gscale, inv_bc1, inv_bc2;
};

// LAMB workspace layout (see ws_workspace_bytes in ws.h).
struct WsLambWs {
    float* rho;        // [T]
    double* norms;     // [T][2]
    float2* partials;  // [R][ntiles]
    // one-launch update: per-tensor arrival counters and ready flags, the ticket counter and the
    // status word (sync_bytes from `count` on are cleared before every launch)
    int* count;        // [T]
    unsigned long long* flag;   // [T] ready words
    unsigned long long* ticket;
    int* status;
    size_t sync_bytes; // from count on
    size_t bytes;      // through the one-launch scratch: what LAMB needs
    float* ghat;       // LARS only: [R][S] summed gradients, 256-byte aligned after the partials
    size_t bytes_lars; // through ghat: what LARS needs
    float* acc;        // Adafactor: [Fi] this step's row / column sums (padded layout)
    double* rsum;      // Adafactor: [T] sum of the new row accumulators, directly after acc
    size_t acc_bytes;  // acc and rsum together: cleared at the start of every step
    // one-kernel Adafactor: arrival counters, ready words and the ticket, directly after rsum and cleared
    // with it (af_sync_bytes from acc on); the status word is the one above
    int *af_count1, *af_countm, *af_count2;        // [T] each
    unsigned long long *af_flagm, *af_flag2;       // [T] each
    unsigned long long* af_ticket;
    size_t af_sync_bytes;
    double2* af_ipart; // [n_afitems] partial sums of w^2 and U^2
    double* af_rfac;   // [af_rows] 1/sqrt(Rv') of the factored tensors' rows
    float* fac;        // Adafactor: [Fi] 1/sqrt factors of V (padded layout)
    float* alpha;      // Adafactor: [T] step sizes
    size_t bytes_af;   // through alpha: what Adafactor needs
};
WsLambWs ws_lamb_layout(const ws_plan* plan, void* workspace);

// Argument checks of LAMB's apply phase for an all-shard call, with no launch (so that a sequence of
// launches can refuse bad arguments before its first one).
ws_status ws_lamb_check_apply_args(const ws_plan* plan, const ws_state* state, const ws_hyper* hyper, const ws_out* out);

// Debug build (-DWS_DEBUG_BOUNDS): before a kernel touches a work item it compares the item's range
// with the extents of the buffers it was given; a range outside them sets a bit in a status word that
// the caller can read (ws_debug_bounds_read) and the item is skipped - no trap, no assert, no access.
enum {
    WS_BOUNDS_STATE = 1,      // w / m / v
    WS_BOUNDS_GRAD = 2,       // a packed gradient buffer
    WS_BOUNDS_OUT = 4,        // the gathered buffer or the stored gradient sum
    WS_BOUNDS_FLAT = 8,       // the flat buffer of ws_pack / ws_unpack
    WS_BOUNDS_SELFTEST = 0x40000000
};
#ifdef WS_DEBUG_BOUNDS
unsigned* ws_bounds_word();   // device address of the status word on the current device, or null
#endif

// error bookkeeping
ws_status ws_cuda_fail(cudaError_t e, const char* what);
ws_status ws_check_launch(const char* what);

static inline bool ws_aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
