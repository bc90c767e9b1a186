// plan.cu -- GPU construction of the standard and node-aware communication
// plans and of the three-block CSR.
//
// Every set of the paper is obtained on the device as a sorted, de-duplicated
// array of packed 64-bit keys:
//   (r, t, j)  r = owner(j) sends column j to the row owner t   Eqs. P, D
//   (n, m, j)  node n sends column j to node m                  Eqs. N, E
//   (t, j)     receive layouts of rank t                        (b_{l->l}, b_{nl->l})
//   (p, s, j)  on_node -> off_node                              Eqs. L0, IL0
//   (q, s, j)  off_node -> on_node                              Eqs. L1, IL1
// built with CUB radix sort / select / run-length encode (library primitives
// for plan time only; the apply path is hand-written).  The per-node-pair
// process assignment T/U (Eqs. T, U and the mapping rule after them, the
// text's variant, or the majority mapping whose per-pair counts are taken on
// the device) is O(node pairs) and runs on the host.  The owner of a row or
// column follows the plan's partition: contiguous blocks (Eq. R) or strided
// (row i on process i mod n_p).  The plan also keeps the matrix split into its
// on_process and remote parts for the overlapped engine.
#include <cub/cub.cuh>

#include <algorithm>
#include <chrono>
#include <cstring>
#include <map>
#include <numeric>

#include "internal.h"

namespace nap {
namespace {

struct NapError {
    int code;
    std::string msg;
};

inline void ck(cudaError_t e, const char *what)
{
    if (e != cudaSuccess) {
        cudaGetLastError();
        throw NapError{e == cudaErrorMemoryAllocation ? NAPSPMV_ERR_OOM : NAPSPMV_ERR_CUDA,
                       std::string(what) + ": " + cudaGetErrorString(e)};
    }
}
#define CK(x) ck((x), #x)

// About what a plan's arrays take, where they are to lie in blocks; else 0.
size_t block_room(const napspmv_plan_t *P);

// Temporaries of one plan build, on one stream: a block given back serves the next
// request that fits it, and all are freed with the build.  About a hundred arrays
// come and go, and each allocation and release of one synchronised the device:
// about 3.4 of 12.4 ms of a 10^6-row 7-point plan (GB300).  A small build takes them
// from one allocation (slab bytes), where some fifty of 3 us and as many releases were a
// tenth of a 64 x 64 grid's plan.
constexpr size_t kSlabMax = 8 << 20;
struct Scratch {
    std::multimap<size_t, void *> idle;
    char *slab = nullptr;
    size_t slab_bytes = 0, used = 0;
    napspmv_plan_t *plan;  // being built
    Scratch *outer = current;
    static thread_local Scratch *current;
    Scratch(napspmv_plan_t *P, size_t slab) : slab_bytes(slab <= kSlabMax ? slab : 0), plan(P)
    {
        current = this;
    }
    ~Scratch()
    {
        trim();
        if (slab) cudaFree(slab);
        current = outer;
    }
    bool in_slab(const void *p) const { return slab && p >= slab && p < slab + slab_bytes; }
    void trim()
    {
        for (auto it = idle.begin(); it != idle.end();) {
            if (in_slab(it->second)) {
                ++it;
            } else {
                cudaFree(it->second);
                it = idle.erase(it);
            }
        }
    }
    void *take(size_t &bytes)
    {
        auto it = idle.lower_bound(bytes);
        if (it != idle.end() && it->first <= 2 * bytes + 4096) {
            void *p = it->second;
            bytes = it->first;
            idle.erase(it);
            return p;
        }
        if (slab_bytes && !slab && cudaMalloc(&slab, slab_bytes) != cudaSuccess) {
            cudaGetLastError();
            slab = nullptr;
            slab_bytes = 0;
        }
        if (used + bytes <= slab_bytes) {
            void *p = slab + used;
            used += bytes;
            return p;
        }
        void *p = nullptr;
        cudaError_t e = cudaMalloc(&p, bytes);
        if (e == cudaErrorMemoryAllocation && !idle.empty()) {
            cudaGetLastError();
            trim();
            e = cudaMalloc(&p, bytes);
        }
        CK(e);
        return p;
    }
};
thread_local Scratch *Scratch::current = nullptr;
// Memory that stays with the plan; idle temporaries make room for it.  The arrays of a
// small or medium plan lie together in a few blocks: fewer allocations, and fewer pages
// for its kernels (a fused apply of 64 x 64 rows, spread among the build's temporaries,
// took 26.3 us for 25.1; GB300).
constexpr size_t kBlockMax = 128 << 20;
template <class T>
cudaError_t device_alloc(T **p, size_t bytes)
{
    Scratch *S = Scratch::current;
    auto get = [&](void **q, size_t b) {
        cudaError_t e = cudaMalloc(q, b);
        if (e == cudaErrorMemoryAllocation && S && !S->idle.empty()) {
            cudaGetLastError();
            S->trim();
            e = cudaMalloc(q, b);
        }
        return e;
    };
    const size_t room = S ? block_room(S->plan) : 0;
    bytes = (bytes + 511) & ~(size_t)511;
    if (room && bytes <= room) {
        auto &B = S->plan->blocks;
        if (B.empty() || B.back().used + bytes > B.back().bytes) {
            const size_t want = B.empty() ? room : std::max(room / 8, bytes);
            void *q = nullptr;
            if (get(&q, want) == cudaSuccess) B.push_back({static_cast<char *>(q), want, 0});
            else cudaGetLastError();
        }
        if (!B.empty() && B.back().used + bytes <= B.back().bytes) {
            *p = reinterpret_cast<T *>(B.back().p + B.back().used);
            B.back().used += bytes;
            return cudaSuccess;
        }
    }
    return get(reinterpret_cast<void **>(p), bytes);
}
// Gives an array of the plan back (one in a block goes with the block).
void device_free(const napspmv_plan_t *P, void *p)
{
    if (!p) return;
    for (const auto &b : P->blocks)
        if (p >= b.p && p < b.p + b.bytes) return;
    cudaFree(p);
}

template <class T>
struct dvec {
    T *p = nullptr;
    int64_t n = 0;
    size_t bytes = 0;  // of a block that came from the scratch
    dvec() = default;
    explicit dvec(int64_t count) { alloc(count); }
    explicit dvec(const std::vector<T> &h) : dvec((int64_t)h.size())
    {
        if (n) CK(cudaMemcpy(p, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice));
    }
    void alloc(int64_t count)
    {
        drop();
        n = count;
        if (count <= 0) return;
        size_t b = (sizeof(T) * (size_t)count + 511) & ~(size_t)511;
        if (Scratch::current) {
            p = static_cast<T *>(Scratch::current->take(b));
            bytes = b;
        } else {
            CK(device_alloc(&p, b));
        }
    }
    void drop()
    {
        if (p && bytes && Scratch::current) Scratch::current->idle.emplace(bytes, p);
        else if (p) cudaFree(p);
        p = nullptr;
        bytes = 0;
    }
    ~dvec() { drop(); }
    void swap(dvec &o)
    {
        std::swap(p, o.p);
        std::swap(n, o.n);
        std::swap(bytes, o.bytes);
    }
    dvec(const dvec &) = delete;
    dvec &operator=(const dvec &) = delete;
};

template <class T>
T *upload(const std::vector<T> &h)
{
    T *d = nullptr;
    size_t bytes = sizeof(T) * std::max<size_t>(h.size(), 1);
    CK(device_alloc(&d, bytes));
    if (!h.empty()) CK(cudaMemcpy(d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice));
    return d;
}

constexpr uint64_t SENT = ~0ull;

inline int bits_for(int64_t maxval)  // bits to hold 0..maxval
{
    int b = 1;
    while (b < 63 && (int64_t(1) << b) <= maxval) b++;
    return b;
}

// Row partition: contiguous blocks of Eq. R (first N mod n_p ranks one row
// longer), or strided (row i on rank i mod n_p, Sec. 5).
struct Part {
    int64_t q, rem, big, np;
    bool strided;
    __host__ __device__ int64_t owner(int64_t j) const
    {
        if (strided) return j % np;
        return j < big ? j / (q + 1) : rem + (j - big) / q;
    }
    // rows of rank r, and its k-th row
    __host__ __device__ int64_t rows(int64_t r) const { return q + (r < rem ? 1 : 0); }
    __host__ __device__ int64_t row(int64_t r, int64_t k) const
    {
        return strided ? r + k * np : start(r) + k;
    }
    // position of row i among its rank's rows
    __host__ __device__ int64_t local(int64_t i) const
    {
        return strided ? i / np : i - start(owner(i));
    }
    // first row of rank r (contiguous blocks only)
    __host__ __device__ int64_t start(int64_t r) const { return r * q + (r < rem ? r : rem); }
};
size_t block_room(const napspmv_plan_t *P)
{
    // some sixty arrays, each on a 512-byte boundary
    const size_t b = (size_t)((P->flags & NAPSPMV_F32_VALUES ? 80 : 60) * P->nnz + 64 * P->n) + (48 << 10);
    return b <= kBlockMax ? b : 0;
}
// About what a build's temporaries take (see Scratch).
size_t slab_for(int64_t n, int64_t nnz) { return (size_t)(64 * nnz + 64 * n); }
Part partition(const napspmv_plan_t *P)
{
    const int64_t q = P->n / P->np, rem = P->n % P->np;
    return Part{q, rem, rem * (q + 1), P->np, (P->flags & NAPSPMV_PARTITION_STRIDED) != 0};
}

inline int blocks_for(int64_t n, int t = 256)
{
    int64_t b = (n + t - 1) / t;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, 1 << 20));
}

// ----------------------------------------------------------------- kernels

__global__ void k_check_rowptr(const int64_t *rp, int64_t n, int64_t nnz, int *bad)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (rp[i + 1] < rp[i]) atomicOr(bad, 1);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && (rp[0] != 0 || rp[n] != nnz)) atomicOr(bad, 1);
}

__global__ void k_row_of(const int64_t *rp, int64_t n, const int32_t *col, int32_t *row_of,
                         int *bad)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        for (int64_t k = rp[i]; k < rp[i + 1]; k++) {
            row_of[k] = (int32_t)i;
            int32_t c = col[k];
            if (c < 0 || c >= n) atomicOr(bad, 2);
        }
    }
}

__global__ void k_pair_keys(const int32_t *row_of, const int32_t *col, int64_t nnz, int jb,
                            uint64_t *keys)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nnz;
         k += (int64_t)gridDim.x * blockDim.x)
        keys[k] = ((uint64_t)row_of[k] << jb) | (uint32_t)col[k];
}

__global__ void k_adjacent_equal(const uint64_t *keys, int64_t n, int *bad)
{
    for (int64_t k = 1 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x)
        if (keys[k] == keys[k - 1]) atomicOr(bad, 4);
}

// Block of every stored entry (Eqs. on_proc, on_node, off_node) and the
// (r, t, j) key of every off-process entry.
__global__ void k_classify(const int32_t *row_of, const int32_t *col, int64_t nnz, Part part,
                           int32_t ppn, int rb, int jb, uint8_t *tag, uint64_t *key,
                           unsigned long long *blk_count)
{
    unsigned long long c[3] = {0, 0, 0};
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nnz;
         k += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = row_of[k], j = col[k];
        int64_t t = part.owner(i), r = part.owner(j);
        uint8_t b = (r == t) ? 0 : ((r / ppn == t / ppn) ? 1 : 2);
        tag[k] = b;
        c[b]++;
        key[k] = b ? (((uint64_t)r << (rb + jb)) | ((uint64_t)t << jb) | (uint64_t)j) : SENT;
    }
    for (int q = 0; q < 3; q++) {
        unsigned long long s = c[q];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0 && s) atomicAdd(&blk_count[q], s);
    }
}

__global__ void k_shift(const uint64_t *in, int64_t n, int sh, uint64_t *out)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x)
        out[k] = in[k] >> sh;
}

__global__ void k_low(const uint64_t *in, int64_t n, uint64_t mask, int32_t *out)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x)
        out[k] = (int32_t)(in[k] & mask);
}

// (r, t, j) -> (t, j)
__global__ void k_rekey_tj(const uint64_t *in, int64_t n, int rb, int jb, uint64_t *out)
{
    uint64_t rmask = (1ull << rb) - 1, jmask = (1ull << jb) - 1;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        uint64_t t = (in[k] >> jb) & rmask;
        out[k] = (t << jb) | (in[k] & jmask);
    }
}

// (r, t, j) -> (node r, node t, j)
__global__ void k_rekey_node(const uint64_t *in, int64_t n, int rb, int jb, int nb, int32_t ppn,
                             uint64_t *out)
{
    uint64_t rmask = (1ull << rb) - 1, jmask = (1ull << jb) - 1;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        uint64_t r = in[k] >> (rb + jb), t = (in[k] >> jb) & rmask;
        out[k] = ((r / ppn) << (nb + jb)) | ((t / ppn) << jb) | (in[k] & jmask);
    }
}

struct NotSent {
    __host__ __device__ bool operator()(uint64_t k) const { return k != SENT; }
};
struct SameNode {
    int rb, jb, ppn;
    bool want;
    __host__ __device__ bool operator()(uint64_t k) const
    {
        uint64_t r = k >> (rb + jb), t = (k >> jb) & ((1ull << rb) - 1);
        return ((r / ppn) == (t / ppn)) == want;
    }
};

__device__ __forceinline__ int64_t lower_bound_i32(const int32_t *a, int64_t n, int32_t x)
{
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (a[mid] < x)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

// Content of g_send (INTER messages in (src, dst) order), its transfer
// destinations in g_recv, the message of every element and the J0 keys.
__global__ void k_fill_gsend(int64_t n_gs, const int64_t *gs_off, int64_t n_msg,
                             const int32_t *msg_pair, const int32_t *msg_src,
                             const int64_t *msg_gr, const int64_t *msg_lo,
                             const int32_t *node_ptr, const int32_t *node_idx, Part part, int rb,
                             int jb, int32_t *gs_j, int32_t *xfer_dst, int32_t *msg_of,
                             uint64_t *j0key)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_gs;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = n_msg - 1;  // last message with gs_off <= e
        while (lo < hi) {
            int64_t mid = (lo + hi + 1) >> 1;
            if (gs_off[mid] <= e)
                lo = mid;
            else
                hi = mid - 1;
        }
        int32_t k = msg_pair[lo];
        int64_t off = e - gs_off[lo];
        int32_t j = node_idx[node_ptr[k] + msg_lo[lo] + off];
        gs_j[e] = j;
        xfer_dst[e] = (int32_t)(msg_gr[lo] + off);
        msg_of[e] = (int32_t)lo;
        int64_t s = msg_src[lo], p = part.owner(j);
        j0key[e] = (p != s) ? (((uint64_t)p << (rb + jb)) | ((uint64_t)s << jb) | (uint64_t)j)
                            : SENT;
    }
}

// Shift of every group of kSendGroup transfer destinations (a warp each).
__global__ void k_xfer_shift(const int32_t *dst, int64_t n, int32_t *shift)
{
    const int lane = threadIdx.x & 31;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g * kSendGroup < n;
         g += warps) {
        const int64_t b = g * kSendGroup;
        const int32_t s = dst[b] - (int32_t)b;
        bool same = true;
        for (int64_t k = b + lane; k < min(n, b + kSendGroup); k += 32)
            same &= dst[k] - (int32_t)k == s;
        same = __all_sync(0xffffffffu, same);
        if (lane == 0) shift[g] = same ? s : kMixed;
    }
}

__global__ void k_pack_src(int64_t n_gs, const int32_t *gs_j, const int32_t *msg_of,
                           const int32_t *msg_src, const int32_t *lbuf_ptr, const int32_t *lbuf_j,
                           Part part, uint32_t *pack_src, int *bad)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_gs;
         e += (int64_t)gridDim.x * blockDim.x) {
        int32_t j = gs_j[e], s = msg_src[msg_of[e]];
        if (part.owner(j) == s) {
            pack_src[e] = (uint32_t)j;
        } else {
            int64_t b = lbuf_ptr[s], len = lbuf_ptr[s + 1] - b;
            int64_t pos = lower_bound_i32(lbuf_j + b, len, j);
            if (pos >= len || lbuf_j[b + pos] != j) atomicOr(bad, 8);
            pack_src[e] = kFromLbuf | (uint32_t)(b + pos);
        }
    }
}

// Off-node receive entries (t, j): the receiving process q of j's node pair,
// the J1 key (q, t, j) when q != t, and the g_recv position to unpack from.
__global__ void k_unpack_src(int64_t n_bnl, const uint64_t *bnl_keys, int jb, Part part,
                             int32_t ppn, int nb, int64_t n_pairs, const uint64_t *pair_key,
                             const int64_t *pair_piece, const int64_t *piece_lo,
                             const int32_t *piece_dst, const int64_t *piece_gr,
                             const int32_t *node_ptr, const int32_t *node_idx, int rb,
                             uint64_t *j1key, int32_t *unp_src, int *bad)
{
    uint64_t jmask = (1ull << jb) - 1;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_bnl;
         e += (int64_t)gridDim.x * blockDim.x) {
        uint64_t t = bnl_keys[e] >> jb;
        int32_t j = (int32_t)(bnl_keys[e] & jmask);
        uint64_t nj = part.owner(j) / ppn, m = t / ppn;
        uint64_t pk = (nj << nb) | m;
        int64_t lo = 0, hi = n_pairs;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if (pair_key[mid] < pk)
                lo = mid + 1;
            else
                hi = mid;
        }
        if (lo >= n_pairs || pair_key[lo] != pk) {
            atomicOr(bad, 16);
            unp_src[e] = 0;
            j1key[e] = SENT;
            continue;
        }
        int64_t b = node_ptr[lo], len = node_ptr[lo + 1] - b;
        int64_t pos = lower_bound_i32(node_idx + b, len, j);
        if (pos >= len || node_idx[b + pos] != j) atomicOr(bad, 16);
        // the piece of the pair holding position pos: the last one starting at
        // or before it
        int64_t a = pair_piece[lo], z = pair_piece[lo + 1] - 1;
        if (z < a) {
            atomicOr(bad, 16);
            unp_src[e] = 0;
            j1key[e] = SENT;
            continue;
        }
        while (a < z) {
            int64_t mid = (a + z + 1) >> 1;
            if (piece_lo[mid] <= pos)
                a = mid;
            else
                z = mid - 1;
        }
        int64_t q = piece_dst[a];
        j1key[e] = ((int64_t)t != q) ? (((uint64_t)q << (rb + jb)) | (t << jb) | (uint64_t)j)
                                     : SENT;
        unp_src[e] = (int32_t)(piece_gr[a] + pos - piece_lo[a]);
    }
}

// Three-block CSR: every row's entries reordered on_process | on_node |
// off_node (stored order kept inside a block), columns coded by block.
__global__ void k_three_block(const int64_t *rp, int64_t n, const int32_t *col, const double *val,
                              const uint8_t *tag, Part part, const int32_t *bll_ptr,
                              const int32_t *bll_j, const int32_t *bnl_ptr, const int32_t *bnl_j,
                              uint32_t *colenc, double *val_out, float *val32_out,
                              int32_t *split, int32_t *rowptr32, int *bad)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        int64_t t = part.owner(i);
        int64_t pos = rp[i];
        rowptr32[i] = (int32_t)rp[i];
        if (i == n - 1) rowptr32[n] = (int32_t)rp[n];
        for (int blk = 0; blk < 3; blk++) {
            int32_t cnt = 0;
            for (int64_t k = rp[i]; k < rp[i + 1]; k++) {
                if (tag[k] != blk) continue;
                int32_t j = col[k];
                uint32_t enc;
                if (blk == 0) {
                    enc = (uint32_t)j;
                } else {
                    const int32_t *ptr = blk == 1 ? bll_ptr : bnl_ptr;
                    const int32_t *arr = blk == 1 ? bll_j : bnl_j;
                    int64_t b = ptr[t], len = ptr[t + 1] - b;
                    int64_t p = lower_bound_i32(arr + b, len, j);
                    if (p >= len || arr[b + p] != j) atomicOr(bad, 32);
                    enc = ((uint32_t)blk << kBlockShift) | (uint32_t)(b + p);
                }
                colenc[pos] = enc;
                val_out[pos] = val[k];
                if (val32_out) val32_out[pos] = (float)val[k];
                pos++;
                cnt++;
            }
            split[3 * i + blk] = cnt;
        }
    }
}

// Lengths of every row's on_process part (L) and remote part (R); the entry
// after the last row is 0 so that an exclusive scan ends with the totals.
__global__ void k_split_lens(const int32_t *split, int64_t n, int32_t *lenL, int32_t *lenR)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n;
         i += (int64_t)gridDim.x * blockDim.x) {
        lenL[i] = i < n ? split[3 * i] : 0;
        lenR[i] = i < n ? split[3 * i + 1] + split[3 * i + 2] : 0;
    }
}

// Copies each three-block row into its L part (the first split[3i] entries)
// and R part (the rest), keeping the order.
__global__ void k_split_copy(const int32_t *rp, int64_t n, const uint32_t *col, const double *val,
                             const float *val32, const int32_t *rpL, const int32_t *rpR,
                             uint32_t *colL, double *valL, float *val32L, uint32_t *colR,
                             double *valR, float *val32R)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t b = rp[i], nl = rpL[i + 1] - rpL[i], e = rp[i + 1];
        for (int32_t k = 0; k < nl; k++) {
            colL[rpL[i] + k] = col[b + k];
            valL[rpL[i] + k] = val[b + k];
            if (val32L) val32L[rpL[i] + k] = val32[b + k];
        }
        for (int32_t k = b + nl; k < e; k++) {
            const int32_t q = rpR[i] + (k - b - nl);
            colR[q] = col[k];
            valR[q] = val[k];
            if (val32R) val32R[q] = val32[k];
        }
    }
}

// ------------------------------------------------------------ CUB helpers

struct Cub {
    cudaStream_t st = 0;
    dvec<char> tmp;
    dvec<int> num;
    Cub() : num(1) {}
    void *temp(size_t bytes)
    {
        if ((int64_t)bytes > tmp.n) tmp.alloc((int64_t)bytes + 256);
        return tmp.p;
    }
    int64_t read_num()
    {
        int h = 0;
        CK(cudaMemcpy(&h, num.p, sizeof(int), cudaMemcpyDeviceToHost));
        return h;
    }
    template <class F>
    int64_t select(const uint64_t *in, int64_t n, uint64_t *out, F f)
    {
        if (n == 0) return 0;
        size_t b = 0;
        CK(cub::DeviceSelect::If(nullptr, b, in, out, num.p, (int)n, f, st));
        CK(cub::DeviceSelect::If(temp(b), b, in, out, num.p, (int)n, f, st));
        return read_num();
    }
    // sorts keys[0..n) ascending over bits [0, end_bit); alt is scratch
    void sort(uint64_t *keys, uint64_t *alt, int64_t n, int end_bit)
    {
        if (n <= 1) return;
        cub::DoubleBuffer<uint64_t> db(keys, alt);
        size_t b = 0;
        CK(cub::DeviceRadixSort::SortKeys(nullptr, b, db, (int)n, 0, end_bit, st));
        CK(cub::DeviceRadixSort::SortKeys(temp(b), b, db, (int)n, 0, end_bit, st));
        if (db.Current() != keys)
            CK(cudaMemcpyAsync(keys, db.Current(), sizeof(uint64_t) * n,
                               cudaMemcpyDeviceToDevice, st));
    }
    int64_t unique(const uint64_t *in, int64_t n, uint64_t *out)
    {
        if (n == 0) return 0;
        size_t b = 0;
        CK(cub::DeviceSelect::Unique(nullptr, b, in, out, num.p, (int)n, st));
        CK(cub::DeviceSelect::Unique(temp(b), b, in, out, num.p, (int)n, st));
        return read_num();
    }
    // stable sort of (key, row) pairs ascending over bits [0, end_bit); the
    // results end in k and v, k2 and v2 are scratch
    void sort_pairs(dvec<uint64_t> &k, dvec<uint64_t> &k2, dvec<int32_t> &v, dvec<int32_t> &v2,
                    int64_t n, int end_bit)
    {
        if (n <= 1) return;
        cub::DoubleBuffer<uint64_t> dk(k.p, k2.p);
        cub::DoubleBuffer<int32_t> dv(v.p, v2.p);
        size_t b = 0;
        CK(cub::DeviceRadixSort::SortPairs(nullptr, b, dk, dv, (int)n, 0, end_bit, st));
        CK(cub::DeviceRadixSort::SortPairs(temp(b), b, dk, dv, (int)n, 0, end_bit, st));
        if (dk.Current() != k.p) k.swap(k2);
        if (dv.Current() != v.p) v.swap(v2);
    }
    template <class T>
    void exclusive_sum(const T *in, T *out, int64_t n)
    {
        size_t b = 0;
        CK(cub::DeviceScan::ExclusiveSum(nullptr, b, in, out, (int)n, st));
        CK(cub::DeviceScan::ExclusiveSum(temp(b), b, in, out, (int)n, st));
    }
    // runs of equal keys: unique values and lengths, copied to the host
    void rle(const uint64_t *in, int64_t n, std::vector<uint64_t> &uniq,
             std::vector<int32_t> &len)
    {
        uniq.clear();
        len.clear();
        if (n == 0) return;
        // one array: the number of runs, the values, the lengths
        dvec<uint64_t> all(1 + n + (n + 1) / 2);
        int *m_out = reinterpret_cast<int *>(all.p);
        uint64_t *u = all.p + 1;
        int32_t *c = reinterpret_cast<int32_t *>(u + n);
        size_t b = 0;
        CK(cub::DeviceRunLengthEncode::Encode(nullptr, b, in, u, c, m_out, (int)n, st));
        CK(cub::DeviceRunLengthEncode::Encode(temp(b), b, in, u, c, m_out, (int)n, st));
        int m = 0;
        if (n <= 8192) {  // a short list comes whole: three reads were 35 us, this is 17 (GB300)
            std::vector<uint64_t> h(all.n);
            CK(cudaMemcpy(h.data(), all.p, sizeof(uint64_t) * h.size(), cudaMemcpyDeviceToHost));
            memcpy(&m, h.data(), sizeof(m));
            uniq.assign(h.begin() + 1, h.begin() + 1 + m);
            len.resize(m);
            memcpy(len.data(), h.data() + 1 + n, sizeof(int32_t) * m);
            return;
        }
        CK(cudaMemcpy(&m, m_out, sizeof(m), cudaMemcpyDeviceToHost));
        uniq.resize(m);
        len.resize(m);
        CK(cudaMemcpy(uniq.data(), u, sizeof(uint64_t) * m, cudaMemcpyDeviceToHost));
        CK(cudaMemcpy(len.data(), c, sizeof(int32_t) * m, cudaMemcpyDeviceToHost));
    }
};

// Numbers on the device, brought to the host together: every read of its own stops the
// stream, 9 to 16 us (GB300).
struct Picked {
    const void *p[32];
    uint32_t wide;  // bit i: p[i] is of 64 bits
};
__global__ void k_pick(Picked P, int n, int64_t *out)
{
    const int i = threadIdx.x;
    if (i < n)
        out[i] = P.wide >> i & 1 ? *static_cast<const int64_t *>(P.p[i]) : *static_cast<const int32_t *>(P.p[i]);
}
struct Reads {
    Picked P{};
    int64_t *to[32];
    int n = 0;
    void ask(const int64_t *p, int64_t *h)
    {
        P.wide |= 1u << n;
        P.p[n] = p;
        to[n++] = h;
    }
    void ask(const int32_t *p, int64_t *h)
    {
        P.p[n] = p;
        to[n++] = h;
    }
    void take()
    {
        dvec<int64_t> out(32);
        int64_t h[32];
        k_pick<<<1, 32>>>(P, n, out.p);
        CK(cudaGetLastError());
        CK(cudaMemcpy(h, out.p, sizeof(int64_t) * n, cudaMemcpyDeviceToHost));
        for (int i = 0; i < n; i++) *to[i] = h[i];
    }
};

// The windows that sliced rows are sorted in: the blocks of the staged windows
// (nsub blocks of `rows` rows per process), else whole processes, or 1024-row
// blocks of a strided plan.
struct SellCut {
    int32_t nsub = 0, rows = 0;
    __host__ __device__ int64_t count(const Part &part, int64_t n) const
    {
        return nsub ? part.np * nsub : part.strided ? (n + 1023) / 1024 : part.np;
    }
    __device__ int64_t window(const Part &part, int64_t i) const
    {
        if (nsub) return part.owner(i) * nsub + part.local(i) / rows;
        return part.strided ? i / 1024 : part.owner(i);
    }
};

// Sort key of every row for its sliced window: (window, longest first); rows of
// more than kSellLong entries take the window after the last.
constexpr int kSellKeyBits = 9;  // holds kSellLong - length, 0 .. kSellLong
static_assert(kSellLong < (1 << kSellKeyBits), "row lengths of the sliced windows fit the key");
__global__ void k_sell_keys(const int32_t *rp, int64_t n, Part part, SellCut cut, int64_t nwin,
                            uint64_t *key, int32_t *row)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t len = rp[i + 1] - rp[i];
        const uint64_t w = len > kSellLong ? nwin : cut.window(part, i);
        key[i] = (w << kSellKeyBits) | (len > kSellLong ? 0 : kSellLong - len);
        row[i] = (int32_t)i;
    }
}

// A warp per window walks its sorted rows in steps of up to 32: lane l holds
// the length of the l-th row from the chunk's first; the chunk ends before the
// first row of less than half its length.  WRITE: the second pass, which
// writes each chunk's entry and rows at the window's offsets; the first counts
// chunks and slots (window nwin, the long rows, counts none and gives *first_long).
template <bool WRITE>
__global__ void k_sell_cut(const uint64_t *key, const int32_t *row, int64_t n, int64_t nwin,
                           int64_t *nch, int64_t *nsl, const int64_t *och, const int64_t *osl,
                           int2 *info, int32_t *perm, int64_t *first_long)
{
    const int lane = threadIdx.x & 31;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w <= nwin; w += warps) {
        int64_t lim[2];  // the window's rows in the sorted order
        for (int q = 0; q < 2; q++) {
            // 32 probes a step: a load for every factor of 33
            int64_t lo = 0, hi = n;
            const uint64_t x = (uint64_t)(w + q) << kSellKeyBits;
            while (lo < hi) {
                const int64_t step = (hi - lo + 32) / 33, at = lo + (lane + 1) * step - 1;
                const int below = __popc(__ballot_sync(0xffffffffu, at < hi && key[at] < x));
                if (below < 32) hi = min(hi, lo + (below + 1) * step - 1);
                lo += below * step;
            }
            lim[q] = lo;
        }
        if (w == nwin) {
            if (!WRITE && lane == 0) {
                nch[w] = nsl[w] = 0;
                *first_long = lim[0];
            }
            continue;
        }
        int64_t c = WRITE ? och[w] : 0, slot = WRITE ? osl[w] : 0;
        int64_t j = lim[0];
        while (j < lim[1]) {
            const bool in = j + lane < lim[1];
            const int32_t len =
                in ? kSellLong - (int32_t)(key[j + lane] & ((1u << kSellKeyBits) - 1)) : -1;
            const int32_t width = __shfl_sync(0xffffffffu, len, 0);
            const unsigned stop = __ballot_sync(0xffffffffu, !in || 2 * len < width);
            const int nl = stop ? __ffs(stop) - 1 : 32;  // lane 0 never stops
            if (WRITE) {
                if (lane == 0) info[c] = make_int2((int)slot, (width << 6) | nl);
                perm[32 * c + lane] = lane < nl ? row[j + lane] : -1;
            }
            // every chunk starts on an 8-slot boundary (16 bytes of 2-byte columns)
            slot += ((int64_t)width * nl + 7) & ~7ll;
            c++;
            j += nl;
        }
        if (!WRITE && lane == 0) {
            nch[w] = c;
            nsl[w] = slot;
        }
    }
}

// Sliced rows: one warp per chunk copies each lane's row into the chunk's
// column-major slots (slot first + i * lanes + lane holds entry i of the
// lane's row) and pads the slots past the row's end.
__global__ void k_sell_fill(const int32_t *rp, const uint32_t *col, const double *val,
                            const float *val32, const int2 *info, const int32_t *perm,
                            int64_t nch, uint32_t *scol, double *sval, float *sval32)
{
    const int lane = threadIdx.x & 31;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < nch; c += warps) {
        const int2 inf = info[c];
        const int width = inf.y >> 6, nl = inf.y & 63;
        if (lane >= nl) continue;
        const int row = perm[32 * c + lane];
        const int k0 = rp[row], len = rp[row + 1] - k0;
        for (int i = 0; i < width; i++) {
            const int64_t q = (int64_t)inf.x + (int64_t)i * nl + lane;
            const bool in = i < len;
            scol[q] = in ? col[k0 + i] : kSellPad;
            sval[q] = in ? val[k0 + i] : 0.0;
            if (sval32) sval32[q] = in ? val32[k0 + i] : 0.0f;
        }
    }
}

// A sorted, unique key array (prefix << jb | j) becomes a message list whose
// prefix is (src << fb | dst); with fb < 0 the prefix is one process id used
// as both src and dst (the per-process buffer layouts).
// Majority mapping (the alternative named after Eq. U), sending side: for
// node pair k (messages of the NODE list, ascending (src, dst)), how many
// values of E(n,m) each process of n owns.  cnt: [M][ppn].
__global__ void k_major_send(const int32_t *idx, int64_t total, const int64_t *ptr, int64_t M,
                             const int32_t *src_node, Part part, int32_t ppn, int32_t *cnt)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t lo = 0, hi = M - 1;  // the pair k with ptr[k] <= e < ptr[k + 1]
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) / 2;
            if (ptr[mid] <= e) lo = mid;
            else hi = mid - 1;
        }
        const int64_t p = part.owner(idx[e]) - (int64_t)src_node[lo] * ppn;
        atomicAdd(&cnt[lo * ppn + p], 1);
    }
}
// Receiving side: every (t, j) of the off-node receive sets (key t << jb | j)
// is a value of E(owner(j)'s node, t's node) that process t's rows use.
__global__ void k_major_recv(const uint64_t *tj, int64_t n, int jb, const uint64_t *pair_key,
                             int64_t M, int nb, Part part, int32_t ppn, int32_t *cnt, int *bad)
{
    const uint64_t jmask = (1ull << jb) - 1;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = (int64_t)(tj[e] >> jb), j = (int64_t)(tj[e] & jmask);
        const int64_t sn = part.owner(j) / ppn, dn = t / ppn;
        const uint64_t key = ((uint64_t)sn << nb) | (uint64_t)dn;
        int64_t lo = 0, hi = M - 1;
        while (lo < hi) {
            const int64_t mid = (lo + hi) / 2;
            if (pair_key[mid] < key) lo = mid + 1;
            else hi = mid;
        }
        if (M == 0 || pair_key[lo] != key) {
            atomicOr(bad, 64);
            continue;
        }
        atomicAdd(&cnt[lo * ppn + (t - dn * ppn)], 1);
    }
}

void make_list(Cub &cb, const uint64_t *keys, int64_t cnt, int fb, int jb, HostList &L)
{
    L = HostList();
    L.ptr.assign(1, 0);
    if (cnt == 0) return;
    dvec<uint64_t> pre(cnt);
    k_shift<<<blocks_for(cnt), 256, 0, cb.st>>>(keys, cnt, jb, pre.p);
    CK(cudaGetLastError());
    std::vector<uint64_t> u;
    std::vector<int32_t> len;
    cb.rle(pre.p, cnt, u, len);
    L.m = (int64_t)u.size();
    L.total = cnt;
    L.src.resize(L.m);
    L.dst.resize(L.m);
    L.ptr.resize(L.m + 1);
    L.ptr[0] = 0;
    for (int64_t k = 0; k < L.m; k++) {
        if (fb < 0) {
            L.src[k] = L.dst[k] = (int32_t)u[k];
        } else {
            L.src[k] = (int32_t)(u[k] >> fb);
            L.dst[k] = (int32_t)(u[k] & ((1ull << fb) - 1));
        }
        L.ptr[k + 1] = L.ptr[k] + len[k];
    }
    CK(device_alloc(&L.d_idx, sizeof(int32_t) * cnt));
    k_low<<<blocks_for(cnt), 256, 0, cb.st>>>(keys, cnt, (1ull << jb) - 1, L.d_idx);
    CK(cudaGetLastError());
}

// Per-process offsets [np+1] of a per-process layout list (empty ranks too).
std::vector<int32_t> full_ptr(const HostList &L, int32_t np)
{
    std::vector<int32_t> p(np + 1, 0);
    std::vector<int64_t> cnt(np, 0);
    for (int64_t k = 0; k < L.m; k++) cnt[L.src[k]] = L.ptr[k + 1] - L.ptr[k];
    for (int32_t r = 0; r < np; r++) p[r + 1] = (int32_t)(p[r] + cnt[r]);
    return p;
}

// The flaws that kernels found so far, by their bits.
void check(int64_t bad)
{
    static const char *const what[] = {"row_ptr must start at 0, never decrease and end at nnz",
                                       "column index out of range [0, n)",
                                       "an entry (i, j) is stored twice",
                                       "internal: pack source missing from the aggregator buffer",
                                       "internal: off-node column without a node-pair message",
                                       "internal: column missing from its receive buffer",
                                       "internal: off-node receive value without a node pair"};
    for (int i = 0; i < 7; i++)
        if (bad >> i & 1) throw NapError{NAPSPMV_ERR_ARG, what[i]};
}
void check(const dvec<int> &bad)
{
    int h = 0;
    CK(cudaMemcpy(&h, bad.p, sizeof(int), cudaMemcpyDeviceToHost));
    check(h);
}

void host_stats(napspmv_plan_t *P)
{
    napspmv_stats &S = P->stats;
    int64_t np = P->np, ppn = P->ppn;
    std::vector<int64_t> a(4 * np, 0), b(4 * np, 0);
    const HostList &St = P->lists[L_STD];
    for (int64_t k = 0; k < St.m; k++) {
        int64_t len = St.ptr[k + 1] - St.ptr[k];
        bool inter = (St.src[k] / ppn) != (St.dst[k] / ppn);
        S.std_msgs++;
        S.std_vals += len;
        if (inter) {
            S.std_inter_msgs++;
            S.std_inter_vals += len;
            a[4 * St.src[k] + 0]++;
            a[4 * St.src[k] + 1] += len;
        } else {
            S.std_intra_msgs++;
            S.std_intra_vals += len;
            a[4 * St.src[k] + 2]++;
            a[4 * St.src[k] + 3] += len;
        }
        S.std_max_msg_vals = std::max(S.std_max_msg_vals, len);
    }
    const HostList &In = P->lists[L_INTER];
    for (int64_t k = 0; k < In.m; k++) {
        int64_t len = In.ptr[k + 1] - In.ptr[k];
        S.nap_inter_msgs++;
        S.nap_inter_vals += len;
        S.nap_max_inter_msg_vals = std::max(S.nap_max_inter_msg_vals, len);
        b[4 * In.src[k] + 0]++;
        b[4 * In.src[k] + 1] += len;
    }
    int64_t *jm[3] = {&S.j0_msgs, &S.j1_msgs, &S.j2_msgs};
    int64_t *jv[3] = {&S.j0_vals, &S.j1_vals, &S.j2_vals};
    const int lk[3] = {L_J0, L_J1, L_J2};
    for (int q = 0; q < 3; q++) {
        const HostList &J = P->lists[lk[q]];
        for (int64_t k = 0; k < J.m; k++) {
            int64_t len = J.ptr[k + 1] - J.ptr[k];
            (*jm[q])++;
            (*jv[q]) += len;
            b[4 * J.src[k] + 2]++;
            b[4 * J.src[k] + 3] += len;
        }
    }
    S.nap_intra_msgs = S.j0_msgs + S.j1_msgs + S.j2_msgs;
    S.nap_intra_vals = S.j0_vals + S.j1_vals + S.j2_vals;
    for (int64_t r = 0; r < np; r++) {
        S.std_max_inter_msgs_proc = std::max(S.std_max_inter_msgs_proc, a[4 * r + 0]);
        S.std_max_inter_vals_proc = std::max(S.std_max_inter_vals_proc, a[4 * r + 1]);
        S.std_max_intra_msgs_proc = std::max(S.std_max_intra_msgs_proc, a[4 * r + 2]);
        S.std_max_intra_vals_proc = std::max(S.std_max_intra_vals_proc, a[4 * r + 3]);
        S.nap_max_inter_msgs_proc = std::max(S.nap_max_inter_msgs_proc, b[4 * r + 0]);
        S.nap_max_inter_vals_proc = std::max(S.nap_max_inter_vals_proc, b[4 * r + 1]);
        S.nap_max_intra_msgs_proc = std::max(S.nap_max_intra_msgs_proc, b[4 * r + 2]);
        S.nap_max_intra_vals_proc = std::max(S.nap_max_intra_vals_proc, b[4 * r + 3]);
    }
    S.node_pairs = P->lists[L_NODE].m;
    S.bll_total = P->n_bll;
    S.bnl_total = P->n_bnl;
    S.lbuf_total = P->n_lbuf;
    double N = (double)P->n, nnz = (double)P->nnz;
    S.bytes_csr_f64 = 4.0 * (N + 1) + nnz * 12.0 + 16.0 * N;
    S.bytes_csr_f32 = 4.0 * (N + 1) + nnz * 8.0 + 16.0 * N;
    S.bytes_msg = 20.0 * (double)(P->n_bll + P->n_lbuf + P->n_gs + P->n_bnl) + 20.0 * (double)P->n_gs;
}

// Rows sorted and cut into chunks, a part's or the staged windows'.
//
// One radix sort of (window, length) keys orders every window at once; a warp
// per window then cuts it, 32 rows to a step.  Sorting and cutting on the host
// (a stable sort per window, three parts, and the upload of the row lists) took
// most of a plan build: 41 of 56 ms of a 10^6-row 7-point plan on GB300, against 2.3 of
// 17 ms this way (810 of 1,180 ms of the 2^23-row banded random plan, against 6 of 370).
struct RowCut {
    int64_t n, nwin;
    dvec<uint64_t> key;
    dvec<int32_t> row;
    // per window, first chunk and first slot; the last element of each is the total;
    // then the first long row's position
    dvec<int64_t> off;
    int64_t total[3] = {};  // chunks, slots, rows of at most kSellLong entries
    const int64_t *och() const { return off.p; }
    const int64_t *osl() const { return off.p + nwin + 1; }
    int wblocks() const { return blocks_for(32 * (nwin + 1)); }

    // (the totals are there once `reads` were taken)
    RowCut(Cub &cb, Reads &reads, const int32_t *d_rp, int64_t rows, const Part &part,
           const SellCut &cut = SellCut())
        : n(rows), nwin(cut.count(part, rows)), key(n), row(n), off(2 * (nwin + 1) + 1)
    {
        dvec<uint64_t> key2(n);
        dvec<int32_t> row2(n);
        k_sell_keys<<<blocks_for(n), 256>>>(d_rp, n, part, cut, nwin, key.p, row.p);
        CK(cudaGetLastError());
        cb.sort_pairs(key, key2, row, row2, n, kSellKeyBits + bits_for(nwin));
        dvec<int64_t> cnt(2 * (nwin + 1));
        int64_t *nch = cnt.p, *nsl = cnt.p + nwin + 1;
        k_sell_cut<false><<<wblocks(), 256>>>(key.p, row.p, n, nwin, nch, nsl, nullptr, nullptr,
                                              nullptr, nullptr, off.p + 2 * (nwin + 1));
        CK(cudaGetLastError());
        cb.exclusive_sum(nch, off.p, nwin + 1);
        cb.exclusive_sum(nsl, off.p + nwin + 1, nwin + 1);
        reads.ask(och() + nwin, &total[0]);
        reads.ask(osl() + nwin, &total[1]);
        reads.ask(osl() + nwin + 1, &total[2]);
    }
    RowCut(const RowCut &) = delete;
    // 31-bit slots
    bool fits() const { return total[1] <= (int64_t)INT32_MAX - 1024; }
    // the chunks, and room for their slots
    void chunks(SellPart &S, bool f32, bool columns) const
    {
        S.nch = total[0];
        S.slots = total[1];
        CK(device_alloc(&S.d_info, sizeof(int2) * std::max<int64_t>(S.nch, 1)));
        CK(device_alloc(&S.d_perm, sizeof(int32_t) * 32 * std::max<int64_t>(S.nch, 1)));
        k_sell_cut<true><<<wblocks(), 256>>>(key.p, row.p, n, nwin, nullptr, nullptr, och(), osl(),
                                             S.d_info, S.d_perm, nullptr);
        CK(cudaGetLastError());
        // padded past the last slot: a block's bulk copy is widened to 16 bytes; a value
        // without a column is not used
        const size_t n_slots = (size_t)std::max<int64_t>(S.slots, 1);
        if (columns) {
            CK(device_alloc(&S.d_col, 4 * n_slots + 256));
            CK(cudaMemset(S.d_col, 0xff, 4 * n_slots + 256));  // kSellPad between chunks too
        }
        CK(device_alloc(&S.d_val, 8 * n_slots + 256));
        if (f32) CK(device_alloc(&S.d_val32, 4 * n_slots + 256));
    }
};

void free_sell(const napspmv_plan_t *P, SellPart &S)
{
    void *p[] = {S.d_info, S.d_perm, S.d_col, S.d_val, S.d_val32, S.d_long};
    for (void *q : p) device_free(P, q);
    S = SellPart();
}

// Sliced-row copy of one matrix part (0 whole, 1 local, 2 remote) from its cut CSR
// rows, built on the device.  Windows: the rows of each process (contiguous
// partition) or of each 1024-row block (strided).  Within a window, rows of at
// most kSellLong entries are sorted by count, longest first (ties by row), and
// cut into chunks of up to 32 whose counts are at least half the first one's;
// longer rows are listed apart.  A part whose padded slots would not fit 31-bit
// offsets is left without a sliced copy.
void build_sell(SellPart &S, const RowCut &R, const int32_t *d_rp, const uint32_t *d_col,
                const double *d_val, const float *d_val32)
{
    const int64_t n = R.n;
    if (!R.fits()) {
        S.slots = -1;  // no sliced copy: NAPSPMV_PIPELINE_SELL is refused for this plan
        return;
    }
    R.chunks(S, d_val32 != nullptr, true);
    S.n_long = (int32_t)(n - R.total[2]);
    CK(device_alloc(&S.d_long, sizeof(int32_t) * std::max<int64_t>(S.n_long, 1)));
    if (S.n_long)
        CK(cudaMemcpy(S.d_long, R.row.p + R.total[2], sizeof(int32_t) * S.n_long,
                      cudaMemcpyDeviceToDevice));
    if (S.nch) {
        k_sell_fill<<<blocks_for(32 * S.nch), 256>>>(d_rp, d_col, d_val, d_val32, S.d_info,
                                                     S.d_perm, S.nch, S.d_col, S.d_val,
                                                     S.d_val32);
        CK(cudaGetLastError());
    }
}

// A block takes at most this much shared memory in FP64: four CTAs to an SM.
constexpr int kWinBytes = 56 * 1024;
// Windows of more values per row than this (strided partitions, whose rows share
// few operands) are mostly gathering: 128 rows to a block and two threads to a row
// (strided 101^3 on GB300: 60.8 us per apply, 78 with 256 rows and a thread each).
// Denser ones take 256 rows and a thread each (contiguous 128^3: 42.6 us, 46 with
// 128 rows, 45 with 512, 59 with two threads).
constexpr int kWinSparse = 5;
// Long rows: 512 rows to a block from this many entries on, 256 from that many in a
// plan without FP32 values, else 128, and half of that until there are two blocks to
// an SM.  Larger blocks gather denser windows, smaller ones overlap better (us per
// apply with 128 / 256 / 512 rows on GB300: 10^6 rows of 20 entries 103 / 107 / 120
// (FP32 values 101 / 104 / 117), 4 * 10^6 480 / 449 / 491 (405 / 424 / 482), 2^23
// 1,135 / 1,060 / 948 (839 / 834 / 835)).
constexpr int64_t kWinLong512 = 140000000, kWinLong256 = 36000000;

// One CTA per block of the staged windows.  The positions of a process's full
// window (own rows, b_{l->l}, b_{nl->l}) that the block's rows use are marked in
// a shared-memory bitmap; a position's slot is its rank among the marked ones.
// COUNT: the size of the block's window.  FILL: its sources, and the window slots and
// values of its sliced rows (a warp per chunk).
struct WinGeom {
    Part part;
    SellCut cut;
    int32_t words;  // bitmap words of the largest process window
    const int32_t *bll_ptr, *bnl_ptr;
};
template <bool FILL>
__global__ void k_win_block(const int32_t *rp, const uint32_t *col, WinGeom G, int64_t nblk,
                            int32_t *nsrc, int32_t *stat, const int64_t *och,
                            const int64_t *osrc, const int32_t *bll_j, const int32_t *unp_src,
                            const double *val, const float *val32, SellPart S, uint32_t *src,
                            uint16_t *col16)
{
    extern __shared__ uint32_t bits[];  // [words], then (FILL) marked positions before each word
    __shared__ int warp_sum[8], block_entries;  // 256 threads
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int64_t b = blockIdx.x; b < nblk; b += gridDim.x) {
        const int64_t t = b / G.cut.nsub, sub = b % G.cut.nsub;
        const int32_t own = (int32_t)G.part.rows(t);
        const int32_t l0 = G.bll_ptr[t], nl = G.bll_ptr[t + 1] - l0;
        const int32_t r0 = G.bnl_ptr[t], nr = G.bnl_ptr[t + 1] - r0;
        const int words = (own + nl + nr + 31) / 32;
        auto position = [&](uint32_t c) {  // in the process's full window
            const int32_t k = (int32_t)(c & kIndexMask);
            const uint32_t blkno = c >> kBlockShift;
            if (blkno == 0) return (int32_t)G.part.local(k);
            return blkno == 1 ? own + k - l0 : own + nl + k - r0;
        };
        for (int w = tid; w < words; w += blockDim.x) bits[w] = 0;
        if (tid == 0) block_entries = 0;
        __syncthreads();
        const int32_t k1 = min(own, (int32_t)(sub + 1) * G.cut.rows);
        int longest = 0, entries = 0;
        for (int32_t k = (int32_t)sub * G.cut.rows + warp; k < k1; k += blockDim.x >> 5) {
            const int64_t i = G.part.row(t, k);
            const int32_t s = rp[i], e = rp[i + 1];
            longest = max(longest, e - s);
            entries += e - s;
            for (int32_t q = s + lane; q < e; q += 32) {
                const int32_t f = position(col[q]);
                atomicOr(&bits[f >> 5], 1u << (f & 31));
            }
        }
        __syncthreads();
        // marked positions before this thread's run of words
        const int per = (words + blockDim.x - 1) / blockDim.x;
        const int w0 = min(words, tid * per), w1 = min(words, w0 + per);
        int mine = 0;
        for (int w = w0; w < w1; w++) mine += __popc(bits[w]);
        int incl = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        int before = incl - mine;
        for (int w = 0; w < warp; w++) before += warp_sum[w];
        if (!FILL) {
            if (lane == 0 && longest) atomicMax(&stat[0], longest);
            if (lane == 0 && entries) atomicAdd(&block_entries, entries);
            __syncthreads();
            if (tid == blockDim.x - 1) {
                nsrc[b] = before + mine;
                atomicMax(&stat[1], before + mine);
                atomicMax(&stat[2], block_entries);
            }
        } else {
            uint32_t *pre = bits + G.words;
            const int64_t s0 = osrc[b];
            for (int w = w0; w < w1; w++) {
                pre[w] = before;
                for (uint32_t m = bits[w]; m; m &= m - 1) {
                    const int32_t f = 32 * w + __ffs(m) - 1;
                    src[s0 + before] = f < own        ? (uint32_t)G.part.row(t, f)
                                       : f < own + nl ? kFromNode | (uint32_t)bll_j[l0 + f - own]
                                                      : kFromRecv | (uint32_t)unp_src[r0 + f - own - nl];
                    before++;
                }
            }
            __syncthreads();
            for (int64_t c = och[b] + warp; c < och[b + 1]; c += blockDim.x >> 5) {
                const int2 inf = S.d_info[c];
                const int width = inf.y >> 6, nlane = inf.y & 63;
                if (lane >= nlane) continue;
                const int32_t i = S.d_perm[32 * c + lane], k0 = rp[i], len = rp[i + 1] - k0;
                for (int k = 0; k < width; k++) {
                    const int64_t q = (int64_t)inf.x + (int64_t)k * nlane + lane;
                    if (k >= len) break;  // (the padding is there)
                    const int32_t f = position(col[k0 + k]);
                    col16[q] = (uint16_t)(pre[f >> 5] + __popc(bits[f >> 5] & ((1u << (f & 31)) - 1)));
                    S.d_val[q] = val[k0 + k];
                    if (S.d_val32) S.d_val32[q] = val32[k0 + k];
                }
            }
        }
        __syncthreads();
    }
}

// Source runs of every block (a warp each) from its source list src[osrc ..].
// COUNT: words needed, a multiple of 4.  WRITE: the runs.
template <bool WRITE>
__global__ void k_win_runs(int64_t nblk, const uint32_t *src, const int64_t *osrc,
                           const int32_t *nsrc, int32_t *words, int32_t *most,
                           const int64_t *oword, uint32_t *runs)
{
    const int lane = threadIdx.x & 31;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < nblk; b += warps) {
        const uint32_t *s = src + osrc[b];
        const int n = nsrc[b], tiles = (n + 31) / 32;
        uint32_t *out = WRITE ? runs + oword[b] : nullptr;
        uint32_t r = 0;
        for (int t = 0; t < tiles; t++) {
            const int k = 32 * t + lane;
            const bool start = k < n && (lane == 0 || s[k] != s[k - 1] + 1);
            const uint32_t m = __ballot_sync(0xffffffffu, start);
            if (WRITE) {
                if (lane == 0) {
                    out[2 * t] = m;
                    out[2 * t + 1] = r;
                }
                if (start) out[2 * tiles + r + __popc(m & ((1u << lane) - 1))] = s[k];
            }
            r += __popc(m);
        }
        if (!WRITE && lane == 0) {
            words[b] = (2 * tiles + (int)r + 3) & ~3;
            atomicMax(most, words[b]);
        }
    }
}

__global__ void k_win_blocks(int64_t nblk, const int64_t *och, const int64_t *osl,
                             const int32_t *nsrc, const int32_t *words, const int64_t *oword,
                             int unit, WinBlock *blk)
{
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b >= nblk) return;
    WinBlock B{};
    B.chunk0 = (int32_t)och[b];
    B.chunks = (int32_t)(och[b + 1] - och[b]);
    B.slot0 = (int32_t)osl[b];
    B.slots = (int32_t)(osl[b + 1] - osl[b]);
    B.srcs = nsrc[b];
    B.words = words[b];
    B.word0 = (int32_t)(oword[b] / unit);
    blk[b] = B;
}
__global__ void k_win_slots(int64_t nblk, const int64_t *osl, int32_t *most)
{
    int32_t m = 0;
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < nblk;
         b += (int64_t)gridDim.x * blockDim.x)
        m = max(m, (int32_t)(osl[b + 1] - osl[b]));
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && m) atomicMax(most, m);
}
__global__ void k_widen(const int32_t *in, int64_t n, int64_t *out)  // out[n] = 0
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = i < n ? in[i] : 0;
}

// Far columns: a message's elements are used by one block of rows each and lie far
// apart in x, sorted by index, and what a block takes of them costs a sector per
// value in g_recv.  Sent in the order of the blocks instead, a block's share is
// contiguous.  Messages of which an element has 1.5 users or more on average (near
// columns) keep their order, for the neighbours in index are what the next rows use;
// and so do messages with an element in fewer than 16 of x, whose owners' values then
// share sectors with the index order only.  Us per apply on GB300, FP64, nodes of 2^15
// rows of 20 entries, a fifth of them far, without / with the order, and an element
// in how many: 10^6 rows 102.8 / 105.7 (8), 2 * 10^6 215 / 213 (15), 4 * 10^6
// 449 / 431 (30), 2^23 948 / 900 (64); FP32 values 100.8 / 103.7, 200 / 201, 405 / 399,
// 839 / 810.
constexpr int kFarSpan = 16;

// first[p], uses[p] of g_recv position p: the first block that uses it, how many do
__global__ void k_recv_uses(int64_t nblk, const uint32_t *src, const int64_t *osrc,
                            const int32_t *nsrc, int32_t *first, int32_t *uses)
{
    for (int64_t b = blockIdx.x; b < nblk; b += gridDim.x)
        for (int k = threadIdx.x; k < nsrc[b]; k += blockDim.x) {
            const uint32_t s = src[osrc[b] + k];
            if (!(s & kFromRecv)) continue;
            atomicMin(&first[s & kIndexMask], (int32_t)b);
            atomicAdd(&uses[s & kIndexMask], 1);
        }
}
// Sort keys (message, first user) of the elements of g_send, a CTA per message;
// any: some message is reordered.
__global__ void k_recv_keys(int64_t n_msg, const int64_t *gs_off, const int32_t *gs_j,
                            const int32_t *dst,
                            const int32_t *first, const int32_t *uses, int bits, uint64_t *key,
                            int32_t *val, int *any)
{
    __shared__ unsigned long long all;
    for (int64_t m = blockIdx.x; m < n_msg; m += gridDim.x) {
        const int64_t b = gs_off[m], e = gs_off[m + 1];
        if (threadIdx.x == 0) all = 0;
        __syncthreads();
        unsigned long long sum = 0;
        for (int64_t k = b + threadIdx.x; k < e; k += blockDim.x) sum += uses[dst[k]];
        atomicAdd(&all, sum);
        __syncthreads();
        const bool far = e > b && 2 * all < 3 * (unsigned long long)(e - b) &&
                         gs_j[e - 1] - gs_j[b] >= kFarSpan * (e - b);
        if (far && threadIdx.x == 0) *any = 1;
        for (int64_t k = b + threadIdx.x; k < e; k += blockDim.x) {
            key[k] = ((uint64_t)m << bits) | (uint64_t)(far ? min(first[dst[k]], (1 << bits) - 1) : 0);
            val[k] = (int32_t)k;
        }
        __syncthreads();
    }
}
// Element k of g_send becomes the former element from[k]; its place in g_recv moves along.
__global__ void k_recv_order(int64_t n_gs, const int32_t *from, const int32_t *gs_j,
                             const int32_t *dst, int32_t *send, int32_t *place)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n_gs;
         k += (int64_t)gridDim.x * blockDim.x) {
        send[k] = gs_j[from[k]];
        place[dst[from[k]]] = dst[k];
    }
}
__global__ void k_recv_move(int64_t n, const int32_t *place, uint32_t *src)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x)
        if (src[k] & kFromRecv) src[k] = kFromRecv | (uint32_t)place[src[k] & kIndexMask];
}
// The order in which g_send suits the windows, and their sources moved to it;
// null: the messages stay as they are.
int32_t *order_receives(napspmv_plan_t *P, Cub &cb, int64_t nblk, const int32_t *nsrc,
                        const int64_t *osrc, uint32_t *src, int64_t total, const int64_t *gs_off,
                        int64_t n_msg)
{
    const int64_t n = P->n_gs;
    if (n == 0) return nullptr;
    dvec<int32_t> first(n), uses(n), val(n), val2(n);
    dvec<uint64_t> key(n), key2(n);
    dvec<int> any(1);
    const int bits = bits_for(nblk);
    CK(cudaMemset(first.p, 0x7f, sizeof(int32_t) * n));
    CK(cudaMemset(uses.p, 0, sizeof(int32_t) * n));
    CK(cudaMemset(any.p, 0, sizeof(int)));
    k_recv_uses<<<(int)std::min<int64_t>(nblk, 1 << 20), 256>>>(nblk, src, osrc, nsrc, first.p,
                                                                uses.p);
    CK(cudaGetLastError());
    k_recv_keys<<<(int)std::min<int64_t>(n_msg, 1 << 20), 256>>>(
        n_msg, gs_off, P->lists[L_INTER].d_idx, P->d_xfer_dst, first.p, uses.p, bits, key.p, val.p, any.p);
    CK(cudaGetLastError());
    int some = 0;
    CK(cudaMemcpy(&some, any.p, sizeof(int), cudaMemcpyDeviceToHost));
    if (!some) return nullptr;
    cb.sort_pairs(key, key2, val, val2, n, bits + bits_for(n_msg));
    int32_t *send = nullptr;
    CK(device_alloc(&send, sizeof(int32_t) * n));
    k_recv_order<<<blocks_for(n), 256>>>(n, val.p, P->lists[L_INTER].d_idx, P->d_xfer_dst, send,
                                         first.p);
    CK(cudaGetLastError());
    k_recv_move<<<blocks_for(total), 256>>>(total, first.p, src);
    CK(cudaGetLastError());
    return send;
}

void free_windows(const napspmv_plan_t *P, WinPart &W)
{
    void *p[] = {W.d_col, W.d_blk, W.d_runs, W.d_send};
    for (void *q : p) device_free(P, q);
    free_sell(P, W.rows);
    W = WinPart();
}

// Chooses the block size of the staged windows and builds them, with sliced rows of
// their own: those of the other engines are sorted over a whole process, where a
// 20-entry row's chunks hold 2.3% padding against 15% over 128 rows.  (When the fused
// engine took the windows' rows, a 150,000-row apply went from 50.5 to 59.5 us, a batch
// of eight 100,000-row matrices from 130 to 143, the SpMV step of 10^6 rows from 74 to
// 81.)  No windows: a plan of composed gathers, a row of more than kSellLong entries,
// fewer than 64 rows per process, or blocks that do not fit the shared memory.
void build_windows(napspmv_plan_t *P, Cub &cb)
{
    const int64_t n = P->n;
    const Part part = partition(P);
    int64_t wide = 0;  // largest process window
    for (int64_t t = 0; t < part.np; t++)
        wide = std::max<int64_t>(wide, part.rows(t) + P->h_bll_rank[t + 1] - P->h_bll_rank[t] +
                                           P->h_bnl_rank[t + 1] - P->h_bnl_rank[t]);
    const int64_t words = (wide + 31) / 32;
    const int64_t max_rows = part.rows(0);
    if ((P->flags & NAPSPMV_COMPOSED_GATHERS) || n / part.np < 64 ||
        8 * words > 200 * 1024)
        return;
    struct Made : WinPart {  // freed unless they become the plan's
        const napspmv_plan_t *plan;
        explicit Made(const napspmv_plan_t *P) : plan(P) {}
        ~Made() { free_windows(plan, *this); }
    } W(P);
    WinGeom G{part, SellCut(), (int32_t)words, P->d_bll_rank, P->d_bnl_rank};
    CK(cudaFuncSetAttribute((const void *)k_win_block<false>,
                            cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    CK(cudaFuncSetAttribute((const void *)k_win_block<true>,
                            cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    dvec<int32_t> nsrc, stat(5);  // per block; longest row, largest window, most entries, slots, words
    int64_t nblk = 0;
    int32_t st[5] = {};
    bool fits = false;
    W.long_rows = P->nnz > 12 * n;
    int rows = !W.long_rows                           ? 256
               : P->nnz >= kWinLong512                ? 512
               : P->nnz >= kWinLong256 && !P->d_val32 ? 256
                                                      : 128;
    for (; rows >= 32 && !fits; rows /= 2) {
        G.cut.nsub = (int32_t)((max_rows + rows - 1) / rows);
        G.cut.rows = (int32_t)((max_rows + G.cut.nsub - 1) / G.cut.nsub + 31) & ~31;
        nblk = part.np * G.cut.nsub;
        if (nblk >= (1ll << 31) - 1) break;
        nsrc.alloc(nblk);
        CK(cudaMemset(stat.p, 0, sizeof(st)));
        const int grid = (int)std::min<int64_t>(nblk, 1 << 20);
        k_win_block<false><<<grid, 256, 4 * words>>>(
            P->d_rowptr, P->d_colenc, G, nblk, nsrc.p, stat.p, nullptr, nullptr, nullptr, nullptr,
            nullptr, nullptr, SellPart(), nullptr, nullptr);
        CK(cudaGetLastError());
        CK(cudaMemcpy(st, stat.p, sizeof(st), cudaMemcpyDeviceToHost));
        if (st[0] > kSellLong) return;
        if (W.long_rows) {
            W.threads = 2 * std::max(64, G.cut.rows);
            fits = window_long_bytes(st[1], 8) <= kWinSmem &&
                   (rows <= 64 || nblk >= 2 * (int64_t)P->num_sms);
            continue;
        }
        const bool sparse = st[1] > kWinSparse * G.cut.rows;
        W.threads = sparse ? 2 * G.cut.rows : G.cut.rows;
        fits = window_bytes(st[1], st[2], st[1], 8) <= kWinBytes && !(sparse && rows > 128);
    }
    if (!fits || st[1] >= kWinPad) return;
    dvec<int64_t> wide_n(nblk + 1), osrc(nblk + 1), oword(nblk + 1);
    dvec<int32_t> nword(nblk);
    Reads reads;
    const RowCut R(cb, reads, P->d_rowptr, n, part, G.cut);
    // the most slots a block has, padding included
    k_win_slots<<<blocks_for(nblk), 256>>>(nblk, R.osl(), stat.p + 3);
    CK(cudaGetLastError());
    auto offsets = [&](const int32_t *cnt, dvec<int64_t> &o) {  // their total last
        k_widen<<<blocks_for(nblk + 1), 256>>>(cnt, nblk, wide_n.p);
        CK(cudaGetLastError());
        cb.exclusive_sum(wide_n.p, o.p, nblk + 1);
        return o.p + nblk;
    };
    int64_t total = 0, max_slots = 0;
    reads.ask(offsets(nsrc.p, osrc), &total);
    reads.ask(stat.p + 3, &max_slots);
    reads.take();
    if (!R.fits()) return;
    R.chunks(W.rows, P->d_val32 != nullptr, false);
    if (W.long_rows && total > INT32_MAX) return;
    // every window's sources: a temporary where they become runs
    dvec<uint32_t> list(W.long_rows ? 0 : std::max<int64_t>(total, 1));
    if (W.long_rows) CK(device_alloc(&W.d_runs, sizeof(uint32_t) * std::max<int64_t>(total, 1)));
    uint32_t *src = W.long_rows ? W.d_runs : list.p;
    const size_t slots = (size_t)std::max<int64_t>(W.rows.slots, 1);
    CK(device_alloc(&W.d_col, sizeof(uint16_t) * slots + 256));
    CK(cudaMemset(W.d_col, 0xff, sizeof(uint16_t) * slots + 256));  // kWinPad
    const int grid = (int)std::min<int64_t>(nblk, 1 << 20);
    k_win_block<true><<<grid, 256, 8 * words>>>(
        P->d_rowptr, P->d_colenc, G, nblk, nullptr, nullptr, R.och(), osrc.p,
        P->lists[L_BLL].d_idx, P->d_unp_src, P->d_val, P->d_val32, W.rows, src, W.d_col);
    CK(cudaGetLastError());
    CK(device_alloc(&W.d_blk, sizeof(WinBlock) * nblk));
    const int bgrid = (int)((nblk + 255) / 256);
    if (W.long_rows) {  // plain lists
        k_win_blocks<<<bgrid, 256>>>(nblk, R.och(), R.osl(), nsrc.p, nsrc.p, osrc.p, 1, W.d_blk);
        CK(cudaGetLastError());
        const HostList &In = P->lists[L_INTER];
        const dvec<int64_t> gs_off(In.ptr);
        W.d_send = order_receives(P, cb, nblk, nsrc.p, osrc.p, src, total, gs_off.p, In.m);
    } else {
        const int wgrid = blocks_for(32 * nblk);
        k_win_runs<false><<<wgrid, 256>>>(nblk, src, osrc.p, nsrc.p, nword.p, stat.p + 4, nullptr,
                                            nullptr);
        CK(cudaGetLastError());
        int64_t all = 0, max_words = 0;
        Reads more;
        more.ask(offsets(nword.p, oword), &all);
        more.ask(stat.p + 4, &max_words);
        more.take();
        if (all / 4 > (int64_t)INT32_MAX || window_bytes(st[1], max_slots, max_words, 8) > kWinSmem)
            return;
        W.max_words = (int32_t)max_words;
        CK(device_alloc(&W.d_runs, sizeof(uint32_t) * std::max<int64_t>(all, 1)));
        k_win_runs<true><<<wgrid, 256>>>(nblk, src, osrc.p, nsrc.p, nullptr, nullptr, oword.p,
                                           W.d_runs);
        CK(cudaGetLastError());
        k_win_blocks<<<bgrid, 256>>>(nblk, R.och(), R.osl(), nsrc.p, nword.p, oword.p, 4, W.d_blk);
        CK(cudaGetLastError());
    }
    W.max_src = st[1];
    W.max_slots = (int32_t)max_slots;
    W.blocks = (int32_t)nblk;
    P->win = W;
    static_cast<WinPart &>(W) = WinPart();
}

void build(napspmv_plan_t *P, const napspmv_csr *A)
{
    const int64_t n = A->n, nnz = A->nnz;
    const int32_t np = P->np, ppn = P->ppn, nn = P->nn;
    Cub cb;
    const Part part = partition(P);
    const int jb = bits_for(n - 1), rb = bits_for(np - 1), nb = bits_for(nn - 1);
    if (2 * rb + jb > 63)
        throw NapError{NAPSPMV_ERR_UNSUPPORTED, "N and n_p too large for 64-bit plan keys"};

    // ---- upload and validate the CSR
    dvec<int64_t> rp(n + 1);
    dvec<int32_t> col(nnz);
    dvec<double> val(nnz);
    CK(cudaMemcpy(rp.p, A->row_ptr, sizeof(int64_t) * (n + 1), cudaMemcpyDefault));
    if (nnz) {
        CK(cudaMemcpy(col.p, A->col, sizeof(int32_t) * nnz, cudaMemcpyDefault));
        CK(cudaMemcpy(val.p, A->val, sizeof(double) * nnz, cudaMemcpyDefault));
    }
    dvec<int> bad(1);
    CK(cudaMemset(bad.p, 0, sizeof(int)));
    k_check_rowptr<<<blocks_for(n), 256>>>(rp.p, n, nnz, bad.p);
    CK(cudaGetLastError());
    check(bad);
    dvec<int32_t> row_of(nnz);
    k_row_of<<<blocks_for(n), 256>>>(rp.p, n, col.p, row_of.p, bad.p);
    CK(cudaGetLastError());
    check(bad);

    dvec<uint64_t> keys(nnz), alt(nnz);
    if (nnz) {
        k_pair_keys<<<blocks_for(nnz), 256>>>(row_of.p, col.p, nnz, jb, keys.p);
        CK(cudaGetLastError());
        cb.sort(keys.p, alt.p, nnz, 2 * jb);
        k_adjacent_equal<<<blocks_for(nnz), 256>>>(keys.p, nnz, bad.p);
        CK(cudaGetLastError());
    }

    // ---- classify; the standard plan (Eqs. P, D)
    dvec<uint8_t> tag(nnz);
    dvec<unsigned long long> blk(3);
    CK(cudaMemset(blk.p, 0, 3 * sizeof(unsigned long long)));
    if (nnz) {
        k_classify<<<blocks_for(nnz), 256>>>(row_of.p, col.p, nnz, part, ppn, rb, jb, tag.p,
                                             keys.p, blk.p);
        CK(cudaGetLastError());
    }
    {
        Reads reads;
        int64_t flaw = 0;
        reads.ask(bad.p, &flaw);
        const int64_t *entries = reinterpret_cast<const int64_t *>(blk.p);
        reads.ask(entries, &P->stats.nnz_on_process);
        reads.ask(entries + 1, &P->stats.nnz_on_node);
        reads.ask(entries + 2, &P->stats.nnz_off_node);
        reads.take();
        check(flaw);
    }
    row_of.alloc(0);

    int64_t c = cb.select(keys.p, nnz, alt.p, NotSent{});
    cb.sort(alt.p, keys.p, c, 2 * rb + jb);
    dvec<uint64_t> std_u(c);
    int64_t U = cb.unique(alt.p, c, std_u.p);
    make_list(cb, std_u.p, U, rb, jb, P->lists[L_STD]);

    // on-node part: J2 (Eqs. L2, IL2) and b_{l->l}; off-node part: E, b_{nl->l}
    dvec<uint64_t> on_u(U), off_u(U);
    int64_t n_on = cb.select(std_u.p, U, on_u.p, SameNode{rb, jb, ppn, true});
    int64_t n_off = cb.select(std_u.p, U, off_u.p, SameNode{rb, jb, ppn, false});
    std_u.alloc(0);
    make_list(cb, on_u.p, n_on, rb, jb, P->lists[L_J2]);

    dvec<uint64_t> tj(std::max(n_on, n_off)), tj_alt(std::max(n_on, n_off));
    if (n_on) {
        k_rekey_tj<<<blocks_for(n_on), 256>>>(on_u.p, n_on, rb, jb, tj.p);
        CK(cudaGetLastError());
    }
    cb.sort(tj.p, tj_alt.p, n_on, rb + jb);
    make_list(cb, tj.p, n_on, -1, jb, P->lists[L_BLL]);
    on_u.alloc(0);

    if (n_off) {
        k_rekey_tj<<<blocks_for(n_off), 256>>>(off_u.p, n_off, rb, jb, tj.p);
        CK(cudaGetLastError());
    }
    cb.sort(tj.p, tj_alt.p, n_off, rb + jb);
    dvec<uint64_t> bnl_keys(n_off);
    if (n_off)
        CK(cudaMemcpy(bnl_keys.p, tj.p, sizeof(uint64_t) * n_off, cudaMemcpyDeviceToDevice));
    make_list(cb, tj.p, n_off, -1, jb, P->lists[L_BNL]);

    // node plan (Eqs. N, E)
    if (n_off) {
        k_rekey_node<<<blocks_for(n_off), 256>>>(off_u.p, n_off, rb, jb, nb, ppn, tj.p);
        CK(cudaGetLastError());
    }
    cb.sort(tj.p, tj_alt.p, n_off, 2 * nb + jb);
    dvec<uint64_t> node_u(n_off);
    int64_t n_node = cb.unique(tj.p, n_off, node_u.p);
    make_list(cb, node_u.p, n_node, nb, jb, P->lists[L_NODE]);
    off_u.alloc(0);
    tj.alloc(0);
    tj_alt.alloc(0);

    P->n_bll = P->lists[L_BLL].total;
    P->n_bnl = P->lists[L_BNL].total;
    if (P->n_bll >= (1ll << 30) || P->n_bnl >= (1ll << 30))
        throw NapError{NAPSPMV_ERR_UNSUPPORTED, "receive buffer beyond 2^30 values"};

    // ---- T, U (host; O(node pairs))
    const HostList &ND = P->lists[L_NODE];
    const int64_t M = ND.m;
    P->send_proc.assign(M, 0);
    P->recv_proc.assign(M, 0);
    // processes per pair on each side: 1, or a group when the node is split
    std::vector<int32_t> send_cnt(M, 1), recv_cnt(M, 1);
    {
        auto procs = [&](int64_t node) { return (int64_t)std::min<int64_t>(ppn, np - node * ppn); };
        std::vector<std::vector<int64_t>> out_of(nn), in_of(nn);
        for (int64_t k = 0; k < M; k++) {
            out_of[ND.src[k]].push_back(k);
            in_of[ND.dst[k]].push_back(k);
        }
        auto len = [&](int64_t k) { return ND.ptr[k + 1] - ND.ptr[k]; };
        const bool majority = (P->flags & NAPSPMV_MAP_MAJORITY) != 0;
        if (majority && M > 0) {
            // per pair: the process of n owning the most of E(n,m) sends, the
            // process of m whose rows use the most of it receives (ties: lowest)
            dvec<int32_t> cs(M * ppn), cr(M * ppn);
            CK(cudaMemset(cs.p, 0, sizeof(int32_t) * M * ppn));
            CK(cudaMemset(cr.p, 0, sizeof(int32_t) * M * ppn));
            std::vector<uint64_t> pk(M);
            for (int64_t k = 0; k < M; k++) pk[k] = ((uint64_t)ND.src[k] << nb) | (uint64_t)ND.dst[k];
            const dvec<int64_t> d_ptr(ND.ptr);
            const dvec<int32_t> d_src(ND.src);
            const dvec<uint64_t> d_pk(pk);
            k_major_send<<<blocks_for(ND.total), 256>>>(ND.d_idx, ND.total, d_ptr.p, M, d_src.p,
                                                       part, ppn, cs.p);
            CK(cudaGetLastError());
            if (P->n_bnl > 0) {
                k_major_recv<<<blocks_for(P->n_bnl), 256>>>(bnl_keys.p, P->n_bnl, jb, d_pk.p, M, nb,
                                                           part, ppn, cr.p, bad.p);
                CK(cudaGetLastError());
            }
            check(bad);
            std::vector<int32_t> hs(M * ppn), hr(M * ppn);
            CK(cudaMemcpy(hs.data(), cs.p, sizeof(int32_t) * M * ppn, cudaMemcpyDeviceToHost));
            CK(cudaMemcpy(hr.data(), cr.p, sizeof(int32_t) * M * ppn, cudaMemcpyDeviceToHost));
            for (int64_t k = 0; k < M; k++) {
                int64_t bs = 0, br = 0;
                for (int64_t p = 1; p < procs(ND.src[k]); p++)
                    if (hs[k * ppn + p] > hs[k * ppn + bs]) bs = p;
                for (int64_t p = 1; p < procs(ND.dst[k]); p++)
                    if (hr[k * ppn + p] > hr[k * ppn + br]) br = p;
                P->send_proc[k] = (int32_t)bs;
                P->recv_proc[k] = (int32_t)br;
            }
        }
        for (int64_t x = 0; x < (majority ? 0 : nn); x++) {
            auto &o = out_of[x];
            std::stable_sort(o.begin(), o.end(), [&](int64_t a, int64_t b) {
                if (len(a) != len(b)) return len(a) > len(b);
                return ND.dst[a] < ND.dst[b];
            });
            const int64_t px = procs(x);
            const bool split = (P->flags & NAPSPMV_MAP_SPLIT) != 0;
            // node splitting (the text after Eq. U): fewer partners than
            // processes -> partner k gets px / K (+1 for the first px mod K)
            // consecutive processes, counted up from process 0 when sending
            if (split && (int64_t)o.size() < px) {
                const int64_t K = (int64_t)o.size();
                int64_t first = 0;
                for (int64_t k = 0; k < K; k++) {
                    const int64_t size = px / K + (k < px % K ? 1 : 0);
                    P->send_proc[o[k]] = (int32_t)first;
                    send_cnt[o[k]] = (int32_t)size;
                    first += size;
                }
            } else {
                for (size_t k = 0; k < o.size(); k++) P->send_proc[o[k]] = (int32_t)(k % px);
            }
            auto &i = in_of[x];
            bool text = (P->flags & NAPSPMV_MAP_TEXT) != 0;
            std::stable_sort(i.begin(), i.end(), [&](int64_t a, int64_t b) {
                if (len(a) != len(b)) return text ? len(a) > len(b) : len(a) < len(b);
                return ND.src[a] < ND.src[b];
            });
            // receiving: groups counted down from the last process
            if (split && (int64_t)i.size() < px) {
                const int64_t K = (int64_t)i.size();
                int64_t top = px;
                for (int64_t k = 0; k < K; k++) {
                    const int64_t size = px / K + (k < px % K ? 1 : 0);
                    P->recv_proc[i[k]] = (int32_t)(top - size);
                    recv_cnt[i[k]] = (int32_t)size;
                    top -= size;
                }
            } else {
                for (size_t k = 0; k < i.size(); k++)
                    P->recv_proc[i[k]] = (int32_t)(px - 1 - (int64_t)(k % px));
            }
        }
    }

    // ---- G, I: one message per node pair, in (src, dst) order for g_send and
    // (dst, src) order for g_recv.  With node splitting a pair carries
    // c = max(send group, receive group) messages: piece i of E(n,m) (positions
    // floor(i e / c) .. floor((i + 1) e / c) - 1) from the i-th process of the
    // sending group to the i-th of the receiving group, cyclically; empty
    // pieces are no message.
    struct Msg {
        int32_t pair, src, dst;
        int64_t lo, hi;  // positions in E(n,m)
    };
    std::vector<Msg> msgs;
    msgs.reserve(M);
    std::vector<int64_t> pair_piece(M + 1, 0);  // first message (by pair) of each pair
    for (int64_t k = 0; k < M; k++) {
        const int64_t ns = send_cnt[k], nr = recv_cnt[k], c = std::max(ns, nr);
        const int64_t e = ND.ptr[k + 1] - ND.ptr[k];
        for (int64_t i = 0; i < c; i++) {
            const int64_t lo = i * e / c, hi = (i + 1) * e / c;
            if (hi == lo) continue;
            Msg mg;
            mg.pair = (int32_t)k;
            mg.src = (int32_t)(ND.src[k] * ppn + P->send_proc[k] + i % ns);
            mg.dst = (int32_t)(ND.dst[k] * ppn + P->recv_proc[k] + i % nr);
            mg.lo = lo;
            mg.hi = hi;
            msgs.push_back(mg);
        }
        pair_piece[k + 1] = (int64_t)msgs.size();
    }
    const int64_t NM = (int64_t)msgs.size();
    std::vector<int32_t> sorder(NM), rorder(NM);
    std::iota(sorder.begin(), sorder.end(), 0);
    std::iota(rorder.begin(), rorder.end(), 0);
    std::sort(sorder.begin(), sorder.end(), [&](int32_t a, int32_t b) {
        return msgs[a].src != msgs[b].src ? msgs[a].src < msgs[b].src : msgs[a].dst < msgs[b].dst;
    });
    std::sort(rorder.begin(), rorder.end(), [&](int32_t a, int32_t b) {
        return msgs[a].dst != msgs[b].dst ? msgs[a].dst < msgs[b].dst : msgs[a].src < msgs[b].src;
    });
    // g_recv offset of every message (indexed by message in pair order)
    std::vector<int64_t> gr_off(NM, 0);
    {
        int64_t o = 0;
        for (int64_t i = 0; i < NM; i++) {
            gr_off[rorder[i]] = o;
            o += msgs[rorder[i]].hi - msgs[rorder[i]].lo;
        }
    }
    // g_send in (src, dst) order: offsets, and per message (in that order) its
    // pair, first position in E(n,m), sender and g_recv offset
    std::vector<int64_t> gs_off(NM + 1, 0), msg_gr(NM), msg_lo(NM);
    std::vector<int32_t> msg_pair(NM), msg_src(NM);
    for (int64_t i = 0; i < NM; i++) {
        const Msg &mg = msgs[sorder[i]];
        gs_off[i + 1] = gs_off[i] + (mg.hi - mg.lo);
        msg_pair[i] = mg.pair;
        msg_src[i] = mg.src;
        msg_gr[i] = gr_off[sorder[i]];
        msg_lo[i] = mg.lo;
    }
    P->n_gs = gs_off[NM];
    if (P->n_gs >= (1ll << 30))
        throw NapError{NAPSPMV_ERR_UNSUPPORTED, "g_send beyond 2^30 values"};
    {
        HostList &In = P->lists[L_INTER];
        In = HostList();
        In.m = NM;
        In.total = P->n_gs;
        In.src.resize(NM);
        In.dst.resize(NM);
        In.ptr = gs_off;
        for (int64_t i = 0; i < NM; i++) {
            In.src[i] = msgs[sorder[i]].src;
            In.dst[i] = msgs[sorder[i]].dst;
        }
    }
    // per pair, its pieces in position order: first position, receiver and
    // g_recv offset (for the off-node receive entries' unpack sources)
    std::vector<int64_t> piece_lo(NM), piece_gr(NM);
    std::vector<int32_t> piece_dst(NM);
    for (int64_t q = 0; q < NM; q++) {
        piece_lo[q] = msgs[q].lo;
        piece_gr[q] = gr_off[q];
        piece_dst[q] = msgs[q].dst;
    }
    std::vector<int32_t> node_ptr32(M + 1);
    for (int64_t k = 0; k <= M; k++) node_ptr32[k] = (int32_t)ND.ptr[k];
    const dvec<int64_t> d_gs_off(gs_off), d_msg_gr(msg_gr), d_msg_lo(msg_lo);
    const dvec<int32_t> d_msg_pair(msg_pair), d_msg_src(msg_src), d_node_ptr(node_ptr32);

    const int64_t ngs = P->n_gs;
    dvec<int32_t> msg_of(ngs);
    dvec<uint64_t> j0key(ngs), j0alt(ngs);
    if (ngs) {
        CK(device_alloc(&P->lists[L_INTER].d_idx, sizeof(int32_t) * ngs));
        CK(device_alloc(&P->d_xfer_dst, sizeof(int32_t) * ngs));
        k_fill_gsend<<<blocks_for(ngs), 256>>>(ngs, d_gs_off.p, NM, d_msg_pair.p, d_msg_src.p,
                                              d_msg_gr.p, d_msg_lo.p, d_node_ptr.p, ND.d_idx,
                                              part, rb, jb, P->lists[L_INTER].d_idx,
                                              P->d_xfer_dst, msg_of.p, j0key.p);
        CK(cudaGetLastError());
    }

    if (ngs) {
        const int64_t groups = (ngs + kSendGroup - 1) / kSendGroup;
        CK(device_alloc(&P->d_xfer_shift, sizeof(int32_t) * groups));
        k_xfer_shift<<<blocks_for(32 * groups), 256>>>(P->d_xfer_dst, ngs, P->d_xfer_shift);
        CK(cudaGetLastError());
    }

    // ---- J0 (Eqs. L0, IL0) and the aggregator buffers b_{l->nl}
    int64_t nj0 = cb.select(j0key.p, ngs, j0alt.p, NotSent{});
    cb.sort(j0alt.p, j0key.p, nj0, 2 * rb + jb);
    dvec<uint64_t> j0u(nj0);
    int64_t Uj0 = cb.unique(j0alt.p, nj0, j0u.p);
    make_list(cb, j0u.p, Uj0, rb, jb, P->lists[L_J0]);
    if (Uj0) {
        k_rekey_tj<<<blocks_for(Uj0), 256>>>(j0u.p, Uj0, rb, jb, j0key.p);
        CK(cudaGetLastError());
    }
    cb.sort(j0key.p, j0alt.p, Uj0, rb + jb);
    make_list(cb, j0key.p, Uj0, -1, jb, P->lists[L_LBUF]);
    P->n_lbuf = Uj0;
    j0key.alloc(0);
    j0alt.alloc(0);
    j0u.alloc(0);

    std::vector<int32_t> lbuf_ptr = full_ptr(P->lists[L_LBUF], np);
    std::vector<int32_t> bll_ptr = full_ptr(P->lists[L_BLL], np);
    std::vector<int32_t> bnl_ptr = full_ptr(P->lists[L_BNL], np);
    P->h_bll_rank = bll_ptr;
    P->h_bnl_rank = bnl_ptr;
    P->d_bll_rank = upload(bll_ptr);
    P->d_bnl_rank = upload(bnl_ptr);
    const dvec<int32_t> d_lbuf_ptr(lbuf_ptr);
    if (ngs) {
        CK(device_alloc(&P->d_pack_src, sizeof(uint32_t) * ngs));
        k_pack_src<<<blocks_for(ngs), 256>>>(ngs, P->lists[L_INTER].d_idx, msg_of.p, d_msg_src.p,
                                            d_lbuf_ptr.p, P->lists[L_LBUF].d_idx, part,
                                            P->d_pack_src, bad.p);
        CK(cudaGetLastError());
    }
    msg_of.alloc(0);

    // ---- J1 (Eqs. L1_send, IL1) and the unpack sources
    const int64_t nbnl = P->n_bnl;
    std::vector<uint64_t> pair_key(M);
    for (int64_t k = 0; k < M; k++) pair_key[k] = ((uint64_t)ND.src[k] << nb) | ND.dst[k];
    const dvec<uint64_t> d_pair_key(pair_key);
    const dvec<int64_t> d_pair_piece(pair_piece), d_piece_lo(piece_lo), d_piece_gr(piece_gr);
    const dvec<int32_t> d_piece_dst(piece_dst);
    dvec<uint64_t> j1key(nbnl), j1alt(nbnl);
    if (nbnl) {
        CK(device_alloc(&P->d_unp_src, sizeof(int32_t) * nbnl));
        k_unpack_src<<<blocks_for(nbnl), 256>>>(nbnl, bnl_keys.p, jb, part, ppn, nb, M,
                                               d_pair_key.p, d_pair_piece.p, d_piece_lo.p,
                                               d_piece_dst.p, d_piece_gr.p, d_node_ptr.p,
                                               ND.d_idx, rb, j1key.p, P->d_unp_src, bad.p);
        CK(cudaGetLastError());
        check(bad);
    }
    int64_t nj1 = cb.select(j1key.p, nbnl, j1alt.p, NotSent{});
    cb.sort(j1alt.p, j1key.p, nj1, 2 * rb + jb);
    make_list(cb, j1alt.p, nj1, rb, jb, P->lists[L_J1]);
    j1key.alloc(0);
    j1alt.alloc(0);
    bnl_keys.alloc(0);

    // ---- three-block CSR
    // padded so that 16-byte bulk copies of a row range may read past the end
    CK(device_alloc(&P->d_rowptr, sizeof(int32_t) * (n + 16)));
    CK(cudaMemset(P->d_rowptr, 0, sizeof(int32_t) * (n + 16)));
    CK(device_alloc(&P->d_colenc, sizeof(uint32_t) * std::max<int64_t>(nnz, 1) + 64));
    CK(device_alloc(&P->d_val, sizeof(double) * std::max<int64_t>(nnz, 1) + 64));
    CK(device_alloc(&P->d_split, sizeof(int32_t) * 3 * n));
    if (P->flags & NAPSPMV_F32_VALUES)
        CK(device_alloc(&P->d_val32, sizeof(float) * std::max<int64_t>(nnz, 1) + 64));
    k_three_block<<<blocks_for(n), 256>>>(rp.p, n, col.p, val.p, tag.p, part, P->d_bll_rank,
                                         P->lists[L_BLL].d_idx, P->d_bnl_rank,
                                         P->lists[L_BNL].d_idx, P->d_colenc, P->d_val,
                                         P->d_val32, P->d_split, P->d_rowptr, bad.p);
    CK(cudaGetLastError());

    // ---- local / remote split
    {
        dvec<int32_t> lenL(n + 1), lenR(n + 1);
        CK(device_alloc(&P->d_rowptrL, sizeof(int32_t) * (n + 16)));
        CK(device_alloc(&P->d_rowptrR, sizeof(int32_t) * (n + 16)));
        CK(cudaMemset(P->d_rowptrL, 0, sizeof(int32_t) * (n + 16)));
        CK(cudaMemset(P->d_rowptrR, 0, sizeof(int32_t) * (n + 16)));
        k_split_lens<<<blocks_for(n + 1), 256>>>(P->d_split, n, lenL.p, lenR.p);
        CK(cudaGetLastError());
        size_t b = 0;
        CK(cub::DeviceScan::ExclusiveSum(nullptr, b, lenL.p, P->d_rowptrL, (int)(n + 1)));
        void *tmp = cb.temp(b);
        CK(cub::DeviceScan::ExclusiveSum(tmp, b, lenL.p, P->d_rowptrL, (int)(n + 1)));
        CK(cub::DeviceScan::ExclusiveSum(tmp, b, lenR.p, P->d_rowptrR, (int)(n + 1)));
        P->nnzL = P->stats.nnz_on_process;
        P->nnzR = nnz - P->nnzL;
        const bool f32 = P->d_val32 != nullptr;
        auto al = [&](int64_t m, size_t sz) {
            void *q = nullptr;
            CK(device_alloc(&q, sz * (size_t)std::max<int64_t>(m, 1) + 64));
            return q;
        };
        P->d_colL = (uint32_t *)al(P->nnzL, 4);
        P->d_valL = (double *)al(P->nnzL, 8);
        P->d_colR = (uint32_t *)al(P->nnzR, 4);
        P->d_valR = (double *)al(P->nnzR, 8);
        if (f32) {
            P->d_val32L = (float *)al(P->nnzL, 4);
            P->d_val32R = (float *)al(P->nnzR, 4);
        }
        k_split_copy<<<blocks_for(n), 256>>>(P->d_rowptr, n, P->d_colenc, P->d_val, P->d_val32,
                                             P->d_rowptrL, P->d_rowptrR, P->d_colL, P->d_valL,
                                             P->d_val32L, P->d_colR, P->d_valR, P->d_val32R);
        CK(cudaGetLastError());
        int lo = 0, hi = 0;
        CK(cudaDeviceGetStreamPriorityRange(&lo, &hi));
        CK(cudaStreamCreateWithPriority(&P->aux, cudaStreamNonBlocking, lo));
        CK(cudaEventCreateWithFlags(&P->ev_fork, cudaEventDisableTiming));
        CK(cudaEventCreateWithFlags(&P->ev_join, cudaEventDisableTiming));
    }

    // sliced-row copies of the whole matrix and of its two split parts
    {
        Reads reads;
        int64_t flaw = 0;
        reads.ask(bad.p, &flaw);
        const RowCut all(cb, reads, P->d_rowptr, n, part), local(cb, reads, P->d_rowptrL, n, part),
            remote(cb, reads, P->d_rowptrR, n, part);
        reads.take();
        check(flaw);
        build_sell(P->sell[0], all, P->d_rowptr, P->d_colenc, P->d_val, P->d_val32);
        build_sell(P->sell[1], local, P->d_rowptrL, P->d_colL, P->d_valL, P->d_val32L);
        build_sell(P->sell[2], remote, P->d_rowptrR, P->d_colR, P->d_valR, P->d_val32R);
    }
    CK(cudaDeviceSynchronize());

    host_stats(P);
}

// The staged windows come last, when the build's temporaries make room for them (see
// device_alloc), and a plan that the memory has room for only without them is one
// without them.
void add_windows(napspmv_plan_t *P)
{
    try {
        Cub cb;
        build_windows(P, cb);
    } catch (const NapError &e) {
        if (e.code != NAPSPMV_ERR_OOM) throw;
        cudaGetLastError();
    }
}

}  // namespace

// Row tiles.  A list's rows are cut into segments (at most kSegment rows, within a
// node's or a process's rows where the list wants that); a warp per segment lays
// tiles one after another, each as many rows as fit tile_rows rows and tile_nnz
// entries (a longer single row alone).  Cutting the seven lists on the host, row by
// row, took 5.1 of 17.6 ms of a 10^6-row 7-point plan, and their three row pointers
// 0.8 ms to bring there; this way 0.47 ms (GB300).
namespace {
constexpr int kSegment = 16384, kStaged = 1024;
struct TileCut {
    const int32_t *rp[kTileLists];
    int32_t rows[kTileLists], cap[kTileLists];
    int64_t segs[kTileLists];   // of every list
    int32_t group[kTileLists];  // processes per unit that tiles stay within; 0: none
    int32_t sub[kTileLists];    // segments per unit
    Part part;
    int64_t n;
};
template <bool WRITE>
__global__ void k_cut_tiles(TileCut C, int32_t *count, const int64_t *off, int32_t *fit, Item *items)
{
    __shared__ int32_t staged[8][kStaged];  // a warp's row pointers: its tiles follow one another
    const int list = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t *rp = C.rp[list];
    const int32_t rows = C.rows[list], cap = C.cap[list];
    int64_t base = 0;  // of this list among all segments
    for (int q = 0; q < list; q++) base += C.segs[q];
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < C.segs[list]; s += warps) {
        int64_t r, e;
        int32_t unit = 0;
        if (C.group[list]) {
            unit = (int32_t)(s / C.sub[list]);
            const int64_t u0 = C.part.start(min((int64_t)unit * C.group[list], C.part.np));
            const int64_t u1 = C.part.start(min((int64_t)(unit + 1) * C.group[list], C.part.np));
            r = min(u1, u0 + s % C.sub[list] * kSegment);
            e = min(u1, r + kSegment);
        } else {
            r = s * kSegment;
            e = min(C.n, r + kSegment);
        }
        int64_t at = WRITE ? off[base + s] : 0;
        int32_t most = 0, tall = 0;
        int64_t s0 = r;  // staged: row pointers s0 .. s0 + kStaged - 1
        auto stage = [&](int64_t from) {
            __syncwarp();
            s0 = from;
            for (int k = lane; k < kStaged; k += 32) staged[warp][k] = rp[min(s0 + k, e)];
            __syncwarp();
        };
        auto ptr = [&](int64_t i) { return i - s0 < kStaged ? staged[warp][i - s0] : rp[i]; };
        if (r < e) stage(r);
        while (r < e) {
            const int32_t limit = (int32_t)min((int64_t)rows, e - r);
            if (r - s0 + limit >= kStaged && r > s0) stage(r);
            const int32_t k0 = ptr(r);
            int32_t m = 0;  // rows of the tile
            for (;;) {
                const int32_t i = m + lane + 1;
                const unsigned ok = __ballot_sync(0xffffffffu, i <= limit && ptr(r + min(i, limit)) - k0 <= cap);
                if (ok == 0xffffffffu) {
                    m += 32;
                    continue;
                }
                m += __ffs(~ok) - 1;  // (the row pointer ascends: a prefix fits)
                break;
            }
            m = max(m, 1);
            const int32_t k1 = ptr(r + m);
            if (WRITE && lane == 0) {
                Item it{};
                it.kind = kSpmv;
                it.b = (int32_t)r;
                it.e = (int32_t)(r + m);
                it.msg = list == kTilesRH ? unit : 0;
                it.k0 = k0;
                it.k1 = k1;
                items[at] = it;
            }
            if (k1 - k0 <= cap) {
                most = max(most, k1 - k0);
                tall = max(tall, m);
            }
            at++;
            r += m;
        }
        if (!WRITE && lane == 0) {
            count[base + s] = (int32_t)at;
            atomicMax(&fit[2 * list], most);
            atomicMax(&fit[2 * list + 1], tall);
        }
    }
}
}  // namespace

int cut_tiles(napspmv_plan_t *P, int32_t tile_rows, int32_t tile_nnz)
{
    try {
        const int64_t n = P->n;
        const bool strided = (P->flags & NAPSPMV_PARTITION_STRIDED) != 0;
        TileCut C{};
        C.part = partition(P);
        C.n = n;
        int64_t all = 0;
        for (int q = 0; q < kTileLists; q++) {
            const bool warp = q == kWarpTiles || q == kWarpTilesL || q == kWarpTilesR;
            C.rp[q] = q == kTilesL || q == kWarpTilesL   ? P->d_rowptrL
                      : q == kTiles || q == kWarpTiles ? P->d_rowptr
                                                       : P->d_rowptrR;
            C.rows[q] = warp ? std::max(1, tile_rows / 8) : tile_rows;
            C.cap[q] = warp ? std::max(32, tile_nnz / 8) : tile_nnz;
            C.segs[q] = (n + kSegment - 1) / kSegment;
            if (q == kTilesRH && strided) C.segs[q] = 0;
            if (!strided && (q == kTiles || q == kTilesRH)) {
                C.group[q] = q == kTiles ? P->ppn : 1;
                const int64_t units = q == kTiles ? P->nn : P->np;
                const int64_t most = std::min<int64_t>(C.group[q], P->np) * C.part.rows(0);
                C.sub[q] = (int32_t)((most + kSegment - 1) / kSegment);
                C.segs[q] = units * C.sub[q];
            }
            all += C.segs[q];
        }
        Cub cb;
        dvec<int32_t> count(all + 1), fit(2 * kTileLists);
        dvec<int64_t> wide(all + 1), off(all + 1);
        CK(cudaMemset(fit.p, 0, sizeof(int32_t) * 2 * kTileLists));
        const int64_t most = *std::max_element(C.segs, C.segs + kTileLists);
        const dim3 grid((unsigned)std::max<int64_t>(1, std::min<int64_t>((most + 7) / 8, 1 << 16)), kTileLists);
        k_cut_tiles<false><<<grid, 256>>>(C, count.p, nullptr, fit.p, nullptr);
        k_widen<<<blocks_for(all + 1), 256>>>(count.p, all, wide.p);
        CK(cudaGetLastError());
        cb.exclusive_sum(wide.p, off.p, all + 1);
        int64_t first[kTileLists + 1], hf[2 * kTileLists], base = 0;
        Reads reads;
        for (int q = 0; q <= kTileLists; q++) {
            reads.ask(off.p + base, &first[q]);
            if (q < kTileLists) base += C.segs[q];
        }
        for (int q = 0; q < 2 * kTileLists; q++) reads.ask(fit.p + q, &hf[q]);
        reads.take();
        Item *d = nullptr;
        CK(device_alloc(&d, sizeof(Item) * std::max<int64_t>(first[kTileLists], 1)));
        k_cut_tiles<true><<<grid, 256>>>(C, nullptr, off.p, nullptr, d);
        const cudaError_t e = cudaStreamSynchronize(0);
        if (e != cudaSuccess) device_free(P, d);
        CK(e);
        ItemSet &S = P->items;
        device_free(P, S.d_all);
        S.d_all = d;
        for (int q = 0; q < kTileLists; q++) {
            auto &L = S.list[q];
            L.d = d + first[q];
            L.n = (int32_t)(first[q + 1] - first[q]);
            // the stage the list needs: its largest tile that is staged at all
            L.fit_nnz = std::min(C.cap[q], (std::max(32, (int32_t)hf[2 * q]) + 15) & ~15);
            L.fit_rows = std::max(1, (int32_t)hf[2 * q + 1]);
        }
        S.tile_rows = tile_rows;
        S.tile_nnz = tile_nnz;
        S.built = true;
    } catch (const NapError &e) {
        set_error(e.code, e.msg);
        return e.code;
    }
    return NAPSPMV_OK;
}

void plan_free(napspmv_plan_t *P)
{
    if (!P) return;
    int cur = 0;
    cudaGetDevice(&cur);
    cudaSetDevice(P->device);
    if (P->ws) {
        ws_free(P->ws);
        delete P->ws;
    }
    for (auto &g : P->graphs) cudaGraphExecDestroy(g.exec);
    for (auto &L : P->lists) device_free(P, L.d_idx);
    void *ptrs[] = {P->d_split, P->d_rowptr, P->d_colenc, P->d_val, P->d_val32, P->d_pack_src,
                    P->d_xfer_dst, P->d_xfer_shift, P->d_unp_src,
                    P->items.d_all,
                    P->d_rowptrL, P->d_rowptrR, P->d_colL, P->d_colR, P->d_valL, P->d_valR,
                    P->d_val32L, P->d_val32R, P->d_bll_rank, P->d_bnl_rank};
    if (P->aux) cudaStreamDestroy(P->aux);
    if (P->ev_fork) cudaEventDestroy(P->ev_fork);
    if (P->ev_join) cudaEventDestroy(P->ev_join);
    for (void *p : ptrs) device_free(P, p);
    for (auto &S : P->sell) free_sell(P, S);
    free_windows(P, P->win);
    for (auto &b : P->blocks) cudaFree(b.p);
    delete P;
    cudaSetDevice(cur);
}

int plan_create(const napspmv_csr *A, int32_t np, int32_t ppn, uint32_t flags,
                napspmv_plan_t **out)
{
    auto t0 = std::chrono::steady_clock::now();
    if (!out) {
        set_error(NAPSPMV_ERR_ARG, "out is NULL");
        return NAPSPMV_ERR_ARG;
    }
    *out = nullptr;
    if (!A || A->n < 1 || A->nnz < 0 || !A->row_ptr || (A->nnz > 0 && (!A->col || !A->val))) {
        set_error(NAPSPMV_ERR_ARG, "invalid CSR descriptor");
        return NAPSPMV_ERR_ARG;
    }
    if (np < 1 || np > A->n || ppn < 1) {
        set_error(NAPSPMV_ERR_ARG, "need 1 <= n_p <= N and ppn >= 1");
        return NAPSPMV_ERR_ARG;
    }
    if (flags & ~(NAPSPMV_F32_VALUES | NAPSPMV_MAP_TEXT | NAPSPMV_PARTITION_STRIDED |
                  NAPSPMV_MAP_MAJORITY | NAPSPMV_COMPOSED_GATHERS | NAPSPMV_MAP_SPLIT)) {
        set_error(NAPSPMV_ERR_ARG, "unknown plan flag");
        return NAPSPMV_ERR_ARG;
    }
    if ((flags & NAPSPMV_MAP_MAJORITY) && (flags & (NAPSPMV_MAP_TEXT | NAPSPMV_MAP_SPLIT))) {
        set_error(NAPSPMV_ERR_ARG, "NAPSPMV_MAP_MAJORITY excludes NAPSPMV_MAP_TEXT and "
                                   "NAPSPMV_MAP_SPLIT");
        return NAPSPMV_ERR_ARG;
    }
    if (A->n >= (1ll << 30) || A->nnz >= (1ll << 31) - 64) {
        set_error(NAPSPMV_ERR_UNSUPPORTED, "N must be < 2^30 and nnz < 2^31");
        return NAPSPMV_ERR_UNSUPPORTED;
    }
    napspmv_plan_t *P = new napspmv_plan_t();
    P->n = A->n;
    P->nnz = A->nnz;
    P->np = np;
    P->ppn = ppn;
    P->nn = (np + ppn - 1) / ppn;
    P->flags = flags;
    try {
        CK(cudaGetDevice(&P->device));
        CK(cudaDeviceGetAttribute(&P->num_sms, cudaDevAttrMultiProcessorCount, P->device));
        Scratch scratch(P, slab_for(A->n, A->nnz));  // outlives every temporary of the build
        build(P, A);
        P->ws = new napspmv_ws_t();
        int rc = ws_alloc(P, P->ws);
        if (rc == NAPSPMV_ERR_OOM) {
            scratch.trim();
            rc = ws_alloc(P, P->ws);
        }
        if (rc) throw NapError{rc, "workspace allocation failed"};
        P->ws->owned_by_plan = true;
        // defaults, measured on GB300 (FP64, per apply):
        //  - staged windows where the plan has them (k_window, k_window_long);
        //    else, or when asked for, by row length:
        //  - rows of more than 12 stored entries on average: the phased engine
        //    with the sliced rows (one lane per row, no shared-memory stage,
        //    chunk groups dealt round robin).  2^23-row banded random workload:
        //    1.71 ms, against 2.18 ms overlapped with sliced rows and 2.00 ms
        //    overlapped with two-lane warp tiles (its SpMV step alone: 0.72 ms
        //    against 1.04 ms);
        //  - shorter rows (the stencils): the overlapped engine with CTA tiles,
        //    one lane per row, 512 rows / 1536 entries (3D 7-point 128^3: 76 us,
        //    against 79 us phased and 89 us overlapped with sliced rows; staged
        //    windows: 40 us).
        // The lane count and tile shape serve the CTA and warp pipelines when an
        // apply asks for them: one lane per row keeps exactly one FP64 FMA per
        // stored entry (GB300's FP64 pipe is the scarce unit); longer rows take
        // more lanes, with 1024-row / 2048-entry tiles.
        double avg = (double)P->nnz / (double)P->n;
        int vec = avg <= 16 ? 1 : avg <= 32 ? 2 : avg <= 96 ? 4 : avg <= 384 ? 16 : 32;
        int rows = 512 / vec;
        int cap = 1536;
        int ctas = 0;  // occupancy maximum
        const bool sell = P->sell[0].slots >= 0 && avg > 12;
        int pipeline = sell ? NAPSPMV_PIPELINE_SELL : NAPSPMV_PIPELINE_CTA;
        int engine = sell ? NAPSPMV_ENGINE_PHASED : NAPSPMV_ENGINE_OVERLAP;
        if (vec > 1) {
            rows = 1024;
            cap = 2048;
        }
        P->defaults.precision = NAPSPMV_PREC_F64;
        P->defaults.engine = engine;
        P->defaults.vec = vec;
        P->defaults.ctas_per_sm = ctas;
        P->defaults.chunk = 2048;
        P->defaults.tile_rows = rows;
        P->defaults.tile_nnz = cap;
        P->defaults.stages = 2;
        P->defaults.pipeline = pipeline;
        P->defaults.halo = NAPSPMV_HALO_ON;
        P->defaults.timeout_ms = 10000;
        P->defaults.debug_stall = 0;
        rc = build_items(P, P->defaults.tile_rows, P->defaults.tile_nnz);
        if (rc) throw NapError{rc, "row-tile construction failed"};
        add_windows(P);
        if ((rc = window_prepare(P))) throw NapError{rc, "staged windows"};
    } catch (const NapError &e) {
        plan_free(P);
        set_error(e.code, e.msg);
        return e.code;
    } catch (const std::bad_alloc &) {
        plan_free(P);
        set_error(NAPSPMV_ERR_OOM, "host allocation failed");
        return NAPSPMV_ERR_OOM;
    }
    P->stats.plan_ms =
        std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    *out = P;
    return NAPSPMV_OK;
}

}  // namespace nap
