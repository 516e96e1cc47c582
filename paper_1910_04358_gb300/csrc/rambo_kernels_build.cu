// rambo_kernels_build.cu -- index construction and batch bookkeeping.
//
//   partition  phi_r(d) for every document and repetition (Section 3.2).
//   prefix     exclusive prefix of the k-mer counts of a batch, so that the
//              k-mers of all items form one flat index space [0, T).
//   register   DocIDs(M[phi_r(d), r]) += d, as bits of the bucket->document
//              bitmaps (Algorithm 2's DocIDs, the "inverted index mapping B
//              buckets to K documents" of Section 5.2).
//   insert     Algorithm 1: every k-mer x of document d sets bits
//              h_1(x)..h_eta(x) of BFU (phi_r(d), r) for every r.  In the
//              bit-sliced layout that is bit r*B+phi_r(d) of position group
//              h_j(x), set with one atomicOr per repetition or 64-bit word.
#include <cooperative_groups.h>

#include "rambo_insert_common.cuh"

namespace rgpu {
namespace {

constexpr uint32_t FULL = 0xffffffffu;

__global__ void k_partition(uint32_t *phi, uint32_t K, uint32_t R, uint32_t B, uint64_t seed) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (uint64_t)K * R) return;
    const uint32_t d = (uint32_t)(i / R), r = (uint32_t)(i % R);
    const uint64_t h = mh_first_word(mh_mix_key((uint64_t)d), (uint32_t)(seed + 1000 + r));
    phi[i] = (uint32_t)(h % B);
}

// The partition of an index folded to Bh buckets: bucket b + Bh's documents
// join bucket b, whatever map they were placed by.
__global__ void k_fold_partition(uint32_t *folded, const uint32_t *phi, uint64_t n, uint32_t Bh) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) folded[i] = phi[i] % Bh;
}

// -------------------------------------------------------------- prefix scan
constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 16;
constexpr uint64_t SCAN_TILE = (uint64_t)SCAN_THREADS * SCAN_ITEMS;

// Count of item i: its k-mers, or (tile > 0) the tiles of `tile` k-mers of
// an item with more than short_max k-mers (0 for shorter items).
struct CountMode {
    uint32_t tile;
    uint32_t short_max;
};

__device__ __forceinline__ uint64_t kmer_count(const uint64_t *begins, const uint64_t *ends,
                                               uint64_t i, uint32_t k, uint64_t limit,
                                               uint32_t *err, CountMode cm) {
    const uint64_t b0 = begins[i], b1 = ends[i];
    if (b1 < b0 || b1 > limit) {
        if (err) atomicOr(err, ERR_OFFSETS);
        return 0;
    }
    const uint64_t L = b1 - b0;
    const uint64_t nk = L >= k ? L - k + 1 : 0;
    if (cm.tile == 0) return nk;
    if (nk <= cm.short_max) return 0;
    if (nk < (1ull << 31)) return ((uint32_t)nk + cm.tile - 1u) / cm.tile;  // tile < 2^25
    return (nk + cm.tile - 1) / cm.tile;
}

// Block-wide exclusive scan of one value per thread (THREADS a multiple of
// 32, at most 1024); returns the prefix and writes the block total to *total.
template <int THREADS = SCAN_THREADS>
__device__ __forceinline__ uint64_t block_exclusive_scan(uint64_t v, uint64_t *total) {
    __shared__ uint64_t warp_sums[THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint64_t y = __shfl_up_sync(FULL, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) warp_sums[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        uint64_t s = lane < THREADS / 32 ? warp_sums[lane] : 0;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint64_t y = __shfl_up_sync(FULL, s, off);
            if (lane >= off) s += y;
        }
        if (lane < THREADS / 32) warp_sums[lane] = s;  // inclusive warp prefix
    }
    __syncthreads();
    const uint64_t before = wid ? warp_sums[wid - 1] : 0;
    *total = warp_sums[THREADS / 32 - 1];
    __syncthreads();
    return before + incl - v;
}

__global__ void __launch_bounds__(SCAN_THREADS)
k_prefix_partial(const uint64_t *begins, const uint64_t *ends, uint64_t n, uint32_t k,
                 uint64_t limit, uint64_t *bsum, uint32_t *err, CountMode cm) {
    const uint64_t base = (uint64_t)blockIdx.x * SCAN_TILE;
    uint64_t s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        const uint64_t i = base + (uint64_t)j * SCAN_THREADS + threadIdx.x;
        if (i < n) s += kmer_count(begins, ends, i, k, limit, err, cm);
    }
    uint64_t total;
    block_exclusive_scan(s, &total);
    if (threadIdx.x == 0) bsum[blockIdx.x] = total;
}

// One block: exclusive scan of the block sums in place; kcum[n] = grand total.
__global__ void __launch_bounds__(SCAN_THREADS)
k_prefix_blocks(uint64_t *bsum, uint64_t nblk, uint64_t *kcum, uint64_t n) {
    uint64_t carry = 0;
    for (uint64_t b0 = 0; b0 < nblk; b0 += SCAN_THREADS) {
        const uint64_t i = b0 + threadIdx.x;
        const uint64_t v = i < nblk ? bsum[i] : 0;
        uint64_t total;
        const uint64_t ex = block_exclusive_scan(v, &total);
        if (i < nblk) bsum[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) kcum[n] = carry;
}

__global__ void __launch_bounds__(SCAN_THREADS)
k_prefix_final(const uint64_t *begins, const uint64_t *ends, uint64_t n, uint32_t k, uint64_t limit,
               const uint64_t *bsum, uint64_t *kcum, CountMode cm) {
    const uint64_t base = (uint64_t)blockIdx.x * SCAN_TILE;
    uint64_t carry = bsum[blockIdx.x];
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        const uint64_t i = base + (uint64_t)j * SCAN_THREADS + threadIdx.x;
        const uint64_t c = i < n ? kmer_count(begins, ends, i, k, limit, nullptr, cm) : 0;
        uint64_t total;
        const uint64_t ex = block_exclusive_scan(c, &total);
        if (i < n) kcum[i] = carry + ex;
        carry += total;
    }
}

// Up to SCAN_ONCE_MAX items: one launch of one cluster of CL blocks, each
// scanning a share of the items; the shares' totals go through distributed
// shared memory.  Clusters past the first fill `fill` with ones: the bucket
// masks of the batch, which would be a launch of their own.  Bound by latency:
// 20,011 items take 6 us (11 with 256 threads a block, 24 in one block walking
// all the tiles); 100,000 took 23 in three launches (partial sums, their scan,
// a second pass).
constexpr uint32_t SCAN1_TILE = 4096;  // items a block scans at a time
constexpr uint64_t SCAN_ONCE_MAX = 32 * SCAN1_TILE;
constexpr uint64_t SCAN_FILL_BYTES = 64 * 1024;  // a fill block's share, at least

template <int CL, int THREADS>
__global__ void __launch_bounds__(THREADS)
k_prefix_once(const uint64_t *begins, const uint64_t *ends, uint64_t n, uint32_t k, uint64_t limit,
              uint64_t *kcum, uint32_t *err, CountMode cm, uint4 *fill, uint64_t fill16) {
    constexpr int ITEMS = SCAN1_TILE / THREADS;
    if (blockIdx.x >= CL) {
        const uint64_t step = (uint64_t)(gridDim.x - CL) * THREADS;
        for (uint64_t i = (uint64_t)(blockIdx.x - CL) * THREADS + threadIdx.x; i < fill16; i += step)
            fill[i] = make_uint4(FULL, FULL, FULL, FULL);
        return;
    }
    __shared__ uint64_t s_cnt[SCAN1_TILE];
    __shared__ uint64_t s_total[CL];  // totals of the shares up to this block's
    uint64_t share = (n + CL - 1) / CL;
    const uint64_t lo = blockIdx.x * share, hi = lo + share < n ? lo + share : n;
    const bool once = share <= SCAN1_TILE;  // the counts stay in shared memory
    uint64_t sum = 0, total = 0, carry = 0;
    if (CL > 1) {
#pragma unroll 4
        for (uint64_t i = lo + threadIdx.x; i < hi; i += THREADS) {
            const uint64_t c = kmer_count(begins, ends, i, k, limit, err, cm);
            if (once) s_cnt[i - lo] = c;
            sum += c;
        }
        block_exclusive_scan<THREADS>(sum, &total);
        namespace cg = cooperative_groups;
        const cg::cluster_group cluster = cg::this_cluster();
        cluster.sync();  // every block runs, so its shared memory may be written
        if (threadIdx.x < CL && threadIdx.x >= blockIdx.x)
            cluster.map_shared_rank(s_total, threadIdx.x)[blockIdx.x] = total;
        cluster.sync();
        for (uint32_t b = 0; b < blockIdx.x; ++b) carry += s_total[b];
    }
    for (uint64_t base = lo; base < hi; base += SCAN1_TILE) {
        if (CL == 1 || !once)
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                const uint32_t t = threadIdx.x + j * THREADS;
                if (base + t < hi) s_cnt[t] = kmer_count(begins, ends, base + t, k, limit, CL == 1 ? err : nullptr, cm);
            }
        __syncthreads();
        const uint64_t i0 = base + (uint64_t)threadIdx.x * ITEMS;
        uint64_t c[ITEMS];
        sum = 0;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            c[j] = i0 + j < hi ? s_cnt[threadIdx.x * ITEMS + j] : 0;
            sum += c[j];
        }
        uint64_t run = carry + block_exclusive_scan<THREADS>(sum, &total);
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            s_cnt[threadIdx.x * ITEMS + j] = run;  // (the scan ended with a barrier)
            run += c[j];
        }
        __syncthreads();
        for (uint32_t t = threadIdx.x; t < SCAN1_TILE && base + t < hi; t += THREADS) kcum[base + t] = s_cnt[t];
        __syncthreads();
        carry += total;
    }
    if (hi == n && lo < n && threadIdx.x == 0) kcum[n] = carry;
}

template <int CL, int THREADS>
cudaError_t launch_prefix_once(const uint64_t *begins, const uint64_t *ends, uint64_t n, uint32_t k, uint64_t limit,
                               uint64_t *kcum, uint32_t *err, CountMode cm, void *fill, size_t fill_bytes,
                               cudaStream_t s) {
    uint64_t fillers = (fill_bytes + SCAN_FILL_BYTES - 1) / SCAN_FILL_BYTES;
    if (fillers > 256) fillers = 256;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(CL + (fillers + CL - 1) / CL * CL));
    cfg.blockDim = dim3(THREADS);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = CL;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = CL > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_prefix_once<CL, THREADS>, begins, ends, n, k, limit, kcum, err, cm,
                              static_cast<uint4 *>(fill), (uint64_t)((fill_bytes + 15) / 16));
}

// ------------------------------------------------------------- registration
__global__ void k_register(const uint32_t *doc_ids, uint64_t n, const uint32_t *phi, uint32_t K,
                           uint32_t R, uint32_t B, uint32_t W, uint32_t *docbits, uint16_t *slots,
                           uint32_t *err) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * R) return;
    const uint64_t item = i / R;
    const uint32_t r = (uint32_t)(i % R);
    const uint32_t d = doc_ids[item];
    if (d >= K) {
        if (r == 0) atomicOr(err, ERR_DOC_RANGE);
        return;
    }
    const uint32_t b = phi[(uint64_t)d * R + r];
    atomicOr(&docbits[((uint64_t)r * B + b) * W + (d >> 5)], 1u << (d & 31));
    if (slots) slots[answer_slot_index(d, r, R)] = (uint16_t)(4 * (r * B + b));
}

// ------------------------------------------------------------------- insert
constexpr int INSERT_THREADS = 256;
// Blocks per resident block: SMs differ in their distance from the memory, so
// even shares of one resident wave wait for the slowest (streaming epoch: 7.51
// ms with 1, 7.43 with 4, 7.32 with 16 and with 64).
constexpr int INSERT_WAVES = 16;

// Each warp walks a contiguous range of the flat k-mer index, 32 k-mers at a
// time; every lane hashes one k-mer, then the warp sets the 32 records of
// each probe together (RecordSetter).  Bound by DRAM once the index outgrows
// L2: every record reads and writes back the lines of its group.
template <int ETA, int KIND>
__global__ void __launch_bounds__(INSERT_THREADS, 1) k_insert(InsertArgs a) {
    const int lane = threadIdx.x & 31;
    const uint64_t T = a.kcum[a.n];
    const uint64_t warp = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const uint64_t nwarps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    uint64_t per = (T + nwarps - 1) / nwarps;
    per = (per + 31) / 32 * 32;
    if (per < 64) per = 64;
    const uint64_t c0 = warp * per;
    if (c0 >= T) return;
    const uint64_t c1 = c0 + per < T ? c0 + per : T;

    // document of the warp's first k-mer (largest i with kcum[i] <= c0)
    uint64_t lo = 0, hi = a.n;
    while (hi - lo > 1) {
        const uint64_t mid = (lo + hi) >> 1;
        if (a.kcum[mid] <= c0) lo = mid;
        else hi = mid;
    }
    const uint64_t i_first = lo;
    RecordSetter<KIND> set(a, lane);

    for (uint32_t jb = 0; jb < a.eta; jb += ETA) {
        uint64_t item = i_first;
        for (uint64_t base = c0; base < c1; base += 32) {
            const uint64_t g = base + lane;
            uint32_t d = NO_DOC;
            uint64_t c = 0;
            if (g < c1) {
                while (a.kcum[item + 1] <= g) ++item;
                d = a.doc_ids[item];
                if (d >= a.K) {
                    d = NO_DOC;
                } else {
                    const uint64_t start = a.offsets[item] + a.base_shift + (g - a.kcum[item]);
                    c = canonical_from_window(base_window(a.packed, a.packed_bytes, start), a.k);
                }
            }
            const uint64_t km = mh_mix_key(c);
#pragma unroll
            for (int e = 0; e < ETA; ++e) {
                if (jb + e >= a.eta) break;  // warp-uniform
                const uint64_t h = mh_first_word(km, a.seed32 + jb + e);
                set(reduce_pos(h, a.m, a.m_inv), d);
            }
        }
    }
}

// The documents' patterns (RecordSetter KIND 1 and 2): word w of document d's
// group bits.
__global__ void k_patterns(unsigned long long *pattern, const uint32_t *phi, uint32_t K, uint32_t R, uint32_t B,
                           uint32_t Gw) {
    const uint32_t words = Gw > 1 ? Gw / 2 : 1;
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (uint64_t)K * words) return;
    const uint64_t d = i / words;
    const uint32_t w = (uint32_t)(i % words);
    unsigned long long v = 0;
    for (uint32_t r = 0; r < R; ++r) {
        const uint32_t bb = r * B + phi[d * R + r];
        if ((bb >> 6) == w) v |= 1ull << (bb & 63);
    }
    if (Gw > 1) pattern[i] = v;
    else reinterpret_cast<uint32_t *>(pattern)[i] = (uint32_t)v;
}

// --------------------------------------------------------------------- fold
// Folding over (Section 5.3, Fig. 5): B -> Bh = B/2.  In position group p,
// repetition r's row of B bits (bits r*B ..) becomes the OR of its two halves,
// stored as the Bh-bit row at bits r*Bh of the new group.  One warp per group:
// the old group is staged in shared memory, lane r builds row r 32 bits at a
// time, and the new words are assembled with shared-memory atomicOr.
constexpr int FOLD_THREADS = 256;
constexpr int FOLD_MAX_WORDS = 128;  // groups up to 512 bytes

__device__ __forceinline__ uint32_t bits_at(const uint32_t *w, uint32_t nwords, uint32_t bit) {
    const uint32_t i = bit >> 5, sh = bit & 31;
    const uint32_t lo = w[i];
    const uint32_t hi = i + 1 < nwords ? w[i + 1] : 0u;
    return sh ? __funnelshift_r(lo, hi, sh) : lo;
}

__global__ void __launch_bounds__(FOLD_THREADS)
k_fold(const uint32_t *old_index, uint32_t old_gw, uint32_t *new_index, uint32_t new_gw, uint64_t m,
       uint32_t B, uint32_t R) {
    __shared__ uint32_t s_old[FOLD_THREADS / 32][FOLD_MAX_WORDS];
    __shared__ uint32_t s_new[FOLD_THREADS / 32][FOLD_MAX_WORDS];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint32_t Bh = B / 2;
    const uint64_t warp = (uint64_t)blockIdx.x * (FOLD_THREADS / 32) + wib;
    const uint64_t nwarps = (uint64_t)gridDim.x * (FOLD_THREADS / 32);
    for (uint64_t p = warp; p < m; p += nwarps) {
        for (uint32_t i = lane; i < old_gw; i += 32) s_old[wib][i] = old_index[p * old_gw + i];
        for (uint32_t i = lane; i < new_gw; i += 32) s_new[wib][i] = 0;
        __syncwarp();
        for (uint32_t r = lane; r < R; r += 32) {
            for (uint32_t c = 0; c < Bh; c += 32) {
                const uint32_t len = Bh - c < 32 ? Bh - c : 32;
                const uint32_t mask = len == 32 ? FULL : ((1u << len) - 1u);
                const uint32_t x = (bits_at(s_old[wib], old_gw, r * B + c) |
                                    bits_at(s_old[wib], old_gw, r * B + Bh + c)) & mask;
                const uint32_t dst = r * Bh + c;
                const uint32_t wi = dst >> 5, sh = dst & 31;
                atomicOr(&s_new[wib][wi], x << sh);
                if (sh && len > 32 - sh) atomicOr(&s_new[wib][wi + 1], x >> (32 - sh));
            }
        }
        __syncwarp();
        for (uint32_t i = lane; i < new_gw; i += 32) new_index[p * new_gw + i] = s_new[wib][i];
        __syncwarp();
    }
}

// new DocBits[r][b] = old[r][b] | old[r][b + Bh]
__global__ void k_fold_docbits(const uint32_t *old_db, uint32_t *new_db, uint32_t B, uint32_t R,
                               uint32_t W) {
    const uint32_t Bh = B / 2;
    const uint64_t total = (uint64_t)R * Bh * W;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t w = (uint32_t)(i % W);
        const uint64_t rb = i / W;
        const uint32_t b = (uint32_t)(rb % Bh), r = (uint32_t)(rb / Bh);
        new_db[i] = old_db[((uint64_t)r * B + b) * W + w] | old_db[((uint64_t)r * B + b + Bh) * W + w];
    }
}

template <typename KernelT>
int blocks_per_sm(KernelT kernel, int threads) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, 0) != cudaSuccess || n < 1)
        n = 1;
    return n;
}

template <int ETA, int KIND>
cudaError_t launch_insert_k(const InsertArgs &a, int sm_count, cudaStream_t s) {
    static int occ = blocks_per_sm(k_insert<ETA, KIND>, INSERT_THREADS);
    uint64_t blocks = (uint64_t)sm_count * occ * INSERT_WAVES;
    // a warp takes 64 k-mers and more: a small batch needs no more blocks than that
    // (a document of 60 bases, 64-byte groups: 36 us with all of them, 30)
    const uint64_t need = (a.max_kmers + INSERT_THREADS * 2 - 1) / (INSERT_THREADS * 2);
    if (a.max_kmers && blocks > need) blocks = need;
    k_insert<ETA, KIND><<<(unsigned)blocks, INSERT_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

template <int ETA>
cudaError_t launch_insert_t(const InsertArgs &a, int sm_count, cudaStream_t s) {
    switch (a.kind) {
        case 0: return launch_insert_k<ETA, 0>(a, sm_count, s);
        case 1: return launch_insert_k<ETA, 1>(a, sm_count, s);
        default: return launch_insert_k<ETA, 2>(a, sm_count, s);
    }
}

}  // namespace

cudaError_t launch_partition(uint32_t *phi, uint32_t K, uint32_t R, uint32_t B, uint64_t seed,
                             cudaStream_t s) {
    const uint64_t n = (uint64_t)K * R;
    k_partition<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(phi, K, R, B, seed);
    return cudaGetLastError();
}

cudaError_t launch_fold_partition(uint32_t *folded, const uint32_t *phi, uint32_t K, uint32_t R, uint32_t Bh,
                                  cudaStream_t s) {
    const uint64_t n = (uint64_t)K * R;
    k_fold_partition<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(folded, phi, n, Bh);
    return cudaGetLastError();
}

size_t kmer_prefix_block_sums(uint64_t n) { return (size_t)((n + SCAN_TILE - 1) / SCAN_TILE); }

int kmer_prefix_launches(uint64_t n) { return n == 0 ? 0 : n <= SCAN_ONCE_MAX ? 1 : 3; }

cudaError_t launch_kmer_prefix(const uint64_t *begins, const uint64_t *ends, uint64_t n, uint32_t k,
                               uint64_t packed_bytes, uint64_t *kcum, uint64_t *block_sums,
                               uint32_t *err, cudaStream_t s, uint32_t tile, uint32_t short_max, void *fill,
                               size_t fill_bytes) {
    const uint64_t limit = packed_bytes * 4;  // bases addressable from the caller's pointer
    const uint64_t nblk = kmer_prefix_block_sums(n);
    if (nblk == 0) return cudaSuccess;
    const CountMode cm{tile, short_max};
    if (n <= SCAN_ONCE_MAX) {
        if (n <= SCAN1_TILE)
            return launch_prefix_once<1, 1024>(begins, ends, n, k, limit, kcum, err, cm, fill, fill_bytes, s);
        return launch_prefix_once<8, 1024>(begins, ends, n, k, limit, kcum, err, cm, fill, fill_bytes, s);
    }
    if (fill_bytes) {
        const cudaError_t e = cudaMemsetAsync(fill, 0xFF, fill_bytes, s);
        if (e != cudaSuccess) return e;
    }
    k_prefix_partial<<<(unsigned)nblk, SCAN_THREADS, 0, s>>>(begins, ends, n, k, limit, block_sums, err, cm);
    k_prefix_blocks<<<1, SCAN_THREADS, 0, s>>>(block_sums, nblk, kcum, n);
    k_prefix_final<<<(unsigned)nblk, SCAN_THREADS, 0, s>>>(begins, ends, n, k, limit, block_sums, kcum, cm);
    return cudaGetLastError();
}

cudaError_t launch_register_docs(const uint32_t *doc_ids, uint64_t n, const uint32_t *phi,
                                 uint32_t K, uint32_t R, uint32_t B, uint32_t W, uint32_t *docbits,
                                 uint32_t *slots, uint32_t *err, cudaStream_t s) {
    const uint64_t total = n * R;
    if (total == 0) return cudaSuccess;
    k_register<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(doc_ids, n, phi, K, R, B, W, docbits,
                                                               reinterpret_cast<uint16_t *>(slots), err);
    return cudaGetLastError();
}

cudaError_t launch_fold(const uint32_t *old_index, uint32_t old_gw, uint32_t *new_index,
                        uint32_t new_gw, uint64_t m, uint32_t B, uint32_t R,
                        const uint32_t *old_db, uint32_t *new_db, uint32_t W, int sm_count,
                        cudaStream_t s) {
    if (old_gw > FOLD_MAX_WORDS || new_gw > FOLD_MAX_WORDS || (B & 1)) return cudaErrorInvalidValue;
    k_fold<<<sm_count * 8, FOLD_THREADS, 0, s>>>(old_index, old_gw, new_index, new_gw, m, B, R);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_fold_docbits<<<sm_count * 4, 256, 0, s>>>(old_db, new_db, B, R, W);
    return cudaGetLastError();
}

uint64_t pattern_bytes(const Geometry &g) {
    if (g.Gw == 1) return (uint64_t)g.K * 4;
    return g.Gw <= g.R && g.Gw <= 64 ? (uint64_t)g.K * (g.Gw / 2) * 8 : 0;
}

cudaError_t launch_patterns(const Geometry &g, unsigned long long *pattern, const uint32_t *phi, cudaStream_t s) {
    const uint64_t n = (uint64_t)g.K * (g.Gw > 1 ? g.Gw / 2 : 1);
    k_patterns<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pattern, phi, g.K, g.R, g.B, g.Gw);
    return cudaGetLastError();
}

cudaError_t launch_insert(const InsertArgs &a, int sm_count, cudaStream_t s) {
    if (a.lanes < 1 || a.lanes > 32) return cudaErrorInvalidValue;  // a turn holds at least one record
    switch (a.eta) {
        case 1: return launch_insert_t<1>(a, sm_count, s);
        case 2: return launch_insert_t<2>(a, sm_count, s);
        case 3: return launch_insert_t<3>(a, sm_count, s);
        default: return launch_insert_t<4>(a, sm_count, s);
    }
}

// ---------------------------------------------------------------------------
// Document-sharded answers (Section 5.3): shard s holds the documents that
// the routing hash sends to it, as local documents 0..K_s-1; the global
// answer of a query is the union over shards of their answers placed at the
// documents' global ids (the shards' documents are disjoint, so this is a
// concatenation in global document order).  One thread per (query, shard
// word): each set bit is ORed into the global row.
namespace {
__global__ void k_merge_shard(uint64_t n, const uint32_t *masks, uint32_t sw, uint32_t sd,
                              const uint32_t *gid, uint32_t *out, uint32_t ow) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * sw) return;
    const uint64_t q = i / sw;
    const uint32_t w = (uint32_t)(i - q * sw);
    uint32_t v = masks[i];
    while (v) {
        const uint32_t j = 32 * w + (uint32_t)(__ffs(v) - 1);
        v &= v - 1;
        if (j >= sd) break;
        const uint32_t d = gid[j];
        if (d / 32 < ow) atomicOr(out + q * ow + d / 32, 1u << (d & 31));
    }
}
}  // namespace

cudaError_t launch_merge_shard(uint64_t n, const uint32_t *shard_masks, uint32_t shard_words,
                               uint32_t shard_docs, const uint32_t *global_ids, uint32_t *out,
                               uint32_t out_words, cudaStream_t s) {
    const uint64_t items = n * shard_words;
    k_merge_shard<<<(unsigned)((items + 255) / 256), 256, 0, s>>>(n, shard_masks, shard_words, shard_docs,
                                                                   global_ids, out, out_words);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Failure-detection check of a bounded device wait: one thread polls an
// mbarrier that nothing ever completes (no arrivals are made), without
// suspending, and gives up after `spins` polls by latching ERR_WAIT.  Nothing
// faults or hangs; the host reads the latched word as RAMBO_ETIMEOUT.
namespace {
__global__ void k_wait_expiry(uint32_t *err, uint64_t spins) {
    __shared__ unsigned long long bar;
    if (threadIdx.x != 0) return;
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(&bar);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(b), "r"(1u) : "memory");
    for (uint64_t i = 0;; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(b), "r"(0u)
            : "memory");
        if (ok) return;
        if (i >= spins) {
            atomicOr(err, ERR_WAIT);
            return;
        }
    }
}
}  // namespace

cudaError_t launch_wait_expiry(uint32_t *err, uint64_t spins, cudaStream_t s) {
    k_wait_expiry<<<1, 32, 0, s>>>(err, spins);
    return cudaGetLastError();
}

}  // namespace rgpu
