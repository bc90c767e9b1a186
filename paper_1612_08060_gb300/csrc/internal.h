// internal.h -- data structures shared by the library's translation units.
//
// A plan holds the three-block CSR, the index arrays of every message step of
// the node-aware algorithm and the work-item list of the fused persistent
// kernel; a workspace holds the receive buffers and dependency counters of one
// in-flight apply.  Nothing here is part of the C ABI (include/napspmv.h).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "../../include/napspmv.h"

namespace nap {

// ------------------------------------------------------------------ errors
void set_error(int code, const std::string &msg);
int cuda_error(cudaError_t e, const char *what);
void count_launch(int64_t n = 1);

#define NAP_CUDA(call)                                            \
    do {                                                          \
        cudaError_t e_ = (call);                                  \
        if (e_ != cudaSuccess) return ::nap::cuda_error(e_, #call); \
    } while (0)

#ifdef __CUDACC__
// Programmatic dependent launch (sm_90 and later).  A kernel launched with the
// programmatic-serialization attribute may become resident while its
// predecessor in the stream drains: griddep_wait() waits, in hardware, until
// the predecessor grid has completed and its writes are visible, and
// griddep_done(), called when a CTA has issued its last work, lets the
// dependent grid start as this grid's CTAs finish (a CTA that exits early
// counts as done).  Without a programmatic predecessor both are no-ops.
__device__ __forceinline__ void griddep_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void griddep_done()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
#endif

// ----------------------------------------------------------- column coding
// A column of the three-block CSR stores its block in the top two bits:
// 0 = on-process (index into v), 1 = on-node (index into b_{l->l}),
// 2 = off-node (index into b_{nl->l}); the low 30 bits are the index.
constexpr uint32_t kBlockShift = 30;
constexpr uint32_t kIndexMask = (1u << 30) - 1;
// A pack source with the top bit set reads the aggregator buffer b_{l->nl},
// otherwise v.
constexpr uint32_t kFromLbuf = 0x80000000u;
// Groups of consecutive elements of g_send whose transfer destinations share one
// shift from their positions; kMixed: they do not.
constexpr int kSendGroup = 128;
constexpr int32_t kMixed = INT32_MIN;

// ------------------------------------------------- row tiles (CTA and warp)
enum ItemKind : int32_t {
    kSpmv = 5,  // rows [b, e) of the three-block SpMV
};

struct Item {
    int32_t kind;
    int32_t b, e;    // row range
    int32_t msg;     // remote tiles cut at process bounds: the process
    int32_t k0, k1;  // stored-entry range [row_ptr[b], row_ptr[e])
    int32_t pad[2];
};

// The tile lists: CTA tiles of the whole matrix (cut within each node's rows), of
// its local and remote parts; warp tiles (at most tile_rows / 8 rows, tile_nnz / 8
// entries) of the three; remote CTA tiles cut at process bounds (Item::msg =
// process), for the remote pass with staged receive buffers.
enum TileList { kTiles = 0, kTilesL, kTilesR, kWarpTiles, kWarpTilesL, kWarpTilesR, kTilesRH, kTileLists };
struct ItemSet {
    bool built = false;
    int32_t tile_rows = 0, tile_nnz = 0;
    Item *d_all = nullptr;  // the lists, one after another
    struct {
        Item *d = nullptr;
        int32_t n = 0;
        // largest staged tile (entries, rows): a stage is sized to what its list
        // needs, not to tile_nnz
        int32_t fit_nnz = 0, fit_rows = 0;
    } list[kTileLists];
};

// --------------------------------------------------------------- plan lists
struct HostList {
    int64_t m = 0, total = 0;
    std::vector<int32_t> src, dst;
    std::vector<int64_t> ptr;
    int32_t *d_idx = nullptr;  // global column indices, device
};

enum ListKind { L_STD = 0, L_NODE, L_INTER, L_J0, L_J1, L_J2, L_BLL, L_BNL, L_LBUF, L_COUNT };

// ------------------------------------------------------- sliced rows (SELL)
// One matrix part (whole, local or remote) in sliced-row form: the rows of
// each process (of each 1024-row block for a strided plan) are sorted by
// stored-entry count, longest first (ties by row), and cut into chunks of up
// to 32 rows whose counts lie within a factor of two of the chunk's first.
// Chunk c stores entry i of its lane l at slot info[c].x + i * lanes + l
// (column-major, so a warp reads consecutive slots); a lane's row shorter
// than the chunk's width is padded with kSellPad columns.  Each row keeps its
// stored entry order, so one lane summing it gives the same bits as the
// one-lane-per-row CSR kernels.  Rows longer than kSellLong entries are listed
// apart and summed by a whole warp from the CSR part.
constexpr uint32_t kSellPad = 0xffffffffu;
constexpr int32_t kSellLong = 256;
struct SellPart {
    int64_t nch = 0, slots = 0;
    int32_t n_long = 0;
    int2 *d_info = nullptr;     // per chunk: first slot, (width << 6) | lanes
    int32_t *d_perm = nullptr;  // 32 per chunk: the row of each lane (-1: none)
    uint32_t *d_col = nullptr;  // block-coded columns, kSellPad in the padding
    double *d_val = nullptr;
    float *d_val32 = nullptr;
    int32_t *d_long = nullptr;  // rows of more than kSellLong entries
};

// ------------------------------------------------------ staged windows
// Each process's rows are cut into blocks of `rows` rows, one CTA each.  A
// block's window lists, once each, the values its rows multiply: own vector
// entries, on-node receives (b_{l->l}) and off-node receives (b_{nl->l}), in
// that order.  The CTA brings the window into shared memory (phase 4, and phase
// 1's on-node part) and sums its sliced rows from there: the windows have sliced
// rows of their own, sorted and cut per block, whose stored entry s multiplies window
// slot col[s].
// Where the window's values come from is kept as runs.  For every 32 slots: a
// mask of the slots that start a run (the first always does) and the index of
// its first run, as two words; after them the source of every run's first slot.
// Stencil windows are a few contiguous pieces, so this is about 13 bytes per 32
// values instead of 128.  Plans of long rows keep a plain list: one source a slot.
constexpr uint16_t kWinPad = 0xffff;      // padding slots, as kSellPad
constexpr uint32_t kFromRecv = 0x80000000u;  // source in g_recv, else in x
constexpr uint32_t kFromNode = 0x40000000u;  // an on-node receive, source in x
struct WinBlock {
    int32_t chunk0, chunks;  // its chunks of the windows' sliced rows
    int32_t slot0, slots;    // its stored-entry slots
    int32_t srcs;            // window slots
    int32_t words, word0;    // its runs: words (a multiple of 4), and the first / 4
                             // (long rows: sources, and the first)
    int32_t pad;
};
struct WinPart {
    int32_t blocks = 0;   // 0: the plan has no windows
    SellPart rows;        // the whole matrix's rows, sorted and cut per block (no d_col, d_long)
    int32_t threads = 0;  // per CTA
    bool long_rows = false;     // rows of more than 12 entries: k_window_long
    int32_t long_ctas[2] = {};  // its CTAs per SM (FP64, FP32)
    int32_t max_src = 0, max_slots = 0, max_words = 0;  // largest block: slots, entry slots, run words
    uint16_t *d_col = nullptr;  // window slot of every slot of `rows`
    WinBlock *d_blk = nullptr;
    uint32_t *d_runs = nullptr;
    int32_t *d_send = nullptr;  // not null: the order of g_send the windows' receives want (order_receives)
};

}  // namespace nap

struct napspmv_ws_s {
    napspmv_plan_t *plan = nullptr;
    int device = 0;
    void *mem = nullptr;  // what the buffers below (but hv, hw) lie in
    double *bll = nullptr, *lbuf = nullptr, *gsend = nullptr, *grecv = nullptr, *bnl = nullptr;
    double *xtmp = nullptr;            // chained-apply intermediate vector
    // FP32 mode of the phased engines: FP32 copies of the chain's vectors, and
    // whether the receive buffers hold FP32 copies (their contents are then
    // read as float arrays)
    float *x32[2] = {nullptr, nullptr};
    int buf_f32 = 0;
    // the staged windows keep the receives in shared memory: what a later
    // napspmv_spmv_step takes them from is the last apply's vector, in xtmp, and
    // g_recv (recv_f32: of FP32 copies).  *state (device) is 1 while the last apply
    // that ran kept its vector, 0 while the receive buffers hold its receives;
    // recv_vector is the same as the host sees it, which it does until the caller
    // captures an apply or a step of this workspace (captured).
    // stepped: a step has taken them on the windows.
    bool recv_vector = false, recv_f32 = false, captured = false, stepped = false;
    int *state = nullptr;  // two words, see k_receives
    double *hv = nullptr, *hw = nullptr;  // staging of napspmv_apply_host
    unsigned long long *ctr = nullptr;  // the fused engine's grid barrier: arrivals, generation
    int *err = nullptr;                 // sticky device status
    bool owned_by_plan = false;
};

struct napspmv_plan_s {
    int device = 0;
    int64_t n = 0, nnz = 0;
    int32_t np = 0, ppn = 0, nn = 0;
    uint32_t flags = 0;
    int num_sms = 0;

    struct Block {  // device memory that arrays of the plan lie in
        char *p;
        size_t bytes, used;
    };
    std::vector<Block> blocks;

    nap::HostList lists[nap::L_COUNT];
    std::vector<int32_t> send_proc, recv_proc;  // per NODE pair
    int32_t *d_split = nullptr;                 // 3 per row

    // three-block CSR
    int32_t *d_rowptr = nullptr;
    uint32_t *d_colenc = nullptr;
    double *d_val = nullptr;
    float *d_val32 = nullptr;

    // the same matrix split in two CSR parts for the overlapped engine: the
    // on_process entries (L, columns index v) and the on_node + off_node
    // entries (R, columns coded by block); each row keeps its stored order
    int64_t nnzL = 0, nnzR = 0;
    int32_t *d_rowptrL = nullptr, *d_rowptrR = nullptr;
    uint32_t *d_colL = nullptr, *d_colR = nullptr;
    double *d_valL = nullptr, *d_valR = nullptr;
    float *d_val32L = nullptr, *d_val32R = nullptr;
    // per-process offsets of b_{l->l} and b_{nl->l} (np + 1 each), host and device
    std::vector<int32_t> h_bll_rank, h_bnl_rank;
    int32_t *d_bll_rank = nullptr, *d_bnl_rank = nullptr;
    cudaStream_t aux = nullptr;  // low-priority stream of the local SpMV
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;

    // sizes of the buffers and index arrays of the message steps
    int64_t n_bll = 0, n_lbuf = 0, n_gs = 0, n_bnl = 0;
    uint32_t *d_pack_src = nullptr;  // [n_gs]
    int32_t *d_xfer_dst = nullptr;   // [n_gs]
    int32_t *d_xfer_shift = nullptr;  // [ceil(n_gs / kSendGroup)]
    int32_t *d_unp_src = nullptr;    // [n_bnl]
    // BLL / LBUF list idx arrays double as the J2 / J0 gather sources.

    // sliced-row copies of the whole matrix, its local part and its remote
    // part (index 0, 1, 2), for NAPSPMV_PIPELINE_SELL; built with the plan
    nap::SellPart sell[3];
    nap::WinPart win;  // staged windows
    int64_t wave_gather[2] = {}, wave_send[2] = {};  // CTAs the GPU holds at once (FP64, FP32)
    // an apply that leaves engine, pipeline and tile options unset runs on the
    // staged windows (until napspmv_set_default_opts names some of them)
    bool auto_window = true;

    nap::ItemSet items;
    // instantiated CUDA graphs of chained phased applies, newest last
    struct GraphEntry {
        const void *v, *w, *ws;
        bool window, keep;
        int32_t reps, prec, vec, tile_rows, tile_nnz, engine, stages, pipeline, ctas_per_sm, halo;
        double scale;
        cudaGraphExec_t exec;
        int64_t kernels;
    };
    std::vector<GraphEntry> graphs;
    napspmv_opts defaults{};
    napspmv_stats stats{};
    napspmv_ws_t *ws = nullptr;  // the plan's own workspace
};

namespace nap {
int cut_tiles(napspmv_plan_t *P, int32_t tile_rows, int32_t tile_nnz);  // of every list
int build_items(napspmv_plan_t *P, int32_t tile_rows, int32_t tile_nnz);
constexpr int kWinSmem = 226 * 1024;  // shared memory of a staged-window CTA, at most
int window_bytes(int64_t srcs, int64_t slots, int64_t words, int vb);  // what one with this block needs
int window_long_bytes(int64_t srcs, int vb);
int window_prepare(napspmv_plan_t *P);
int ws_alloc(napspmv_plan_t *P, napspmv_ws_t *ws);
void ws_free(napspmv_ws_t *ws);
void plan_free(napspmv_plan_t *P);
// Options with every unset field resolved; window: run on the staged windows.
struct Opts : napspmv_opts {
    bool window = false;
    bool batch = false;  // FP64 receive buffers in both precisions, as on the fused engine
};
Opts resolve_opts(const napspmv_plan_t *P, const napspmv_opts *o);
// the fields that name an engine, a pipeline or a tile shape are all unset
bool leaves_path_open(const napspmv_opts &o);
// they are all the same
bool same_path(const napspmv_opts &a, const napspmv_opts &b);
// ERR_ARG / ERR_STATE / ERR_UNSUPPORTED (with the message set) for resolved
// options the plan cannot run, else NAPSPMV_OK
int check_opts(const napspmv_plan_t *P, const napspmv_opts &o);
int apply_batch(int32_t count, napspmv_plan_t *const *plans, napspmv_ws_t *const *ws,
                const double *const *v, double *const *w, const int32_t *reps,
                const double *scale, const napspmv_opts *opts, cudaStream_t s, bool keep = true,
                bool as_batch = false);
// Pieces of an apply for a caller that makes its vector itself (CG): whether
// applies at this precision run on short-row staged windows by default; the
// inter-node messages of several vectors alone (one each for distinct plans or
// workspaces); the windowed SpMVs alone; and where the messages go.
bool runs_on_windows(const napspmv_plan_t *P, int32_t precision);
int send_alone(int count, napspmv_plan_t *const *plans, napspmv_ws_t *const *ws, int32_t precision,
               const double *const *x, cudaStream_t s);
int window_alone(int count, napspmv_plan_t *const *plans, napspmv_ws_t *const *ws, int32_t precision,
                 const double *const *x, double *const *y, cudaStream_t s);
struct SendList {
    const int32_t *j, *dst, *shift;  // see k_send
    void *grecv;
    const int *err;
    int32_t n;
};
SendList send_list(const napspmv_plan_t *P, const napspmv_ws_t *ws);
}  // namespace nap
