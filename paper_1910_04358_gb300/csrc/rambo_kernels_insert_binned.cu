// rambo_kernels_insert_binned.cu -- Algorithm 1's bit setting, binned by
// index region so that its atomics hit L2.
//
// The direct insert ORs every probe's bits into a random line of the index:
// once the index outgrows L2, nearly every atomic misses and costs a DRAM
// read and write of the line.  Here a chunk of the batch's k-mers goes
// through two passes:
//   scatter  every probe (k-mer x, document d, position h_j(x)) becomes one
//            8-byte record (h_j(x), d) appended to the bin of its index
//            region; a CTA stages a tile of 4096 records in shared memory,
//            counts them per bin, reserves each bin's share with one global
//            atomicAdd and writes them out;
//   apply    a persistent grid claims units of records in bin order, so all
//            CTAs work inside one or two regions at a time and the regions
//            stay in L2 while their records set bit r*B + phi_r(d) of group
//            h_j(x) for every r (RecordSetter, as in the direct insert).
// Records past a bin's capacity set their bits during the scatter pass.  OR
// is commutative and idempotent, so the index is bit-identical to the
// direct insert's whatever the order.
#include "rambo_insert_binned.cuh"
#include "rambo_insert_common.cuh"

namespace rgpu {
namespace {

constexpr int IB_THREADS = 256;
constexpr uint32_t IB_UNIT = 2048;     // records per unit of the apply pass
constexpr uint32_t IB_UNIT_MIN = 128;  // ... of a small batch, at least

__device__ __forceinline__ uint32_t record_group(unsigned long long rec) { return (uint32_t)(rec >> IB_DOC_BITS); }
__device__ __forceinline__ uint32_t record_doc(unsigned long long rec) {
    return (uint32_t)(rec & ((1u << IB_DOC_BITS) - 1));
}

// Scatter pass over [f0, f1) of the flat k-mer index: each CTA takes a
// contiguous range in tiles of IB_TILE_RECORDS / ETA k-mers, up to ETA probes
// of each per pass over the hash seeds.  A thread takes consecutive k-mers of
// the tile, so that one load of 96 bases' bits and one document lookup serve
// all of them.  Its positions stay in registers with their ranks in their
// bins (counted in shared memory) until every bin's share is reserved, one
// global atomic per tile and bin; then the records go through shared memory in
// bin order (a counting sort), so that a warp's store covers a few runs of
// consecutive slots instead of 32 scattered records.
// Bound by the issue rate (65% of the slots at three blocks an SM; about 300
// instructions per 32 k-mers, half of them hashing).  10^9 k-mers into 1 GiB:
// 11.1 ms, against 14.5 ms with every record staged with its bin and rank,
// k-mers strided over the threads and stores in slot order; three and five
// blocks an SM take 11.6 and 11.6 ms.
constexpr uint32_t IB_TILE_RECORDS = 4096;

// s_sorted (8 bytes a record); s_cnt, s_base, s_pre (4 a bin)
constexpr size_t scatter_smem() { return (size_t)IB_TILE_RECORDS * 8 + (size_t)IB_MAX_BINS * 12; }

// Exclusive prefix of n <= IB_MAX_BINS counts, in place, by the whole CTA;
// returns the total to every thread.
__device__ uint32_t ib_block_scan(uint32_t *v, uint32_t n) {
    __shared__ uint32_t warp_tot[IB_THREADS / 32];
    constexpr uint32_t PER = IB_MAX_BINS / IB_THREADS;
    const uint32_t b0 = threadIdx.x * PER;
    uint32_t sum = 0;
#pragma unroll
    for (uint32_t i = 0; i < PER; ++i) sum += b0 + i < n ? v[b0 + i] : 0u;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) warp_tot[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        uint32_t x = lane < IB_THREADS / 32 ? warp_tot[lane] : 0u;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        if (lane < IB_THREADS / 32) warp_tot[lane] = x;
    }
    __syncthreads();
    uint32_t run = (wid ? warp_tot[wid - 1] : 0u) + incl - sum;
    const uint32_t total = warp_tot[IB_THREADS / 32 - 1];
#pragma unroll
    for (uint32_t i = 0; i < PER; ++i) {
        if (b0 + i < n) {
            const uint32_t x = v[b0 + i];
            v[b0 + i] = run;
            run += x;
        }
    }
    __syncthreads();
    return total;
}

// The 96 bits from base t on, t + i in bits 2i, 2i + 1 (bytes at or past
// nbytes read as zero).
__device__ __forceinline__ void window96(const uint8_t *p, uint64_t nbytes, uint64_t t, uint32_t (&y)[3]) {
    const uint64_t w = t >> 4;
    uint32_t v[4];
    if (w * 4 + 16 <= nbytes) {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = __ldg(reinterpret_cast<const uint32_t *>(p) + w + i);
    } else {
        for (int i = 0; i < 4; ++i) {
            v[i] = 0;
            for (int c = 0; c < 4; ++c)
                if ((w + i) * 4 + c < nbytes) v[i] |= (uint32_t)__ldg(p + (w + i) * 4 + c) << (8 * c);
        }
    }
    const uint32_t sh = (uint32_t)(t & 15) * 2;
#pragma unroll
    for (int i = 0; i < 3; ++i) y[i] = __funnelshift_r(v[i], v[i + 1], sh);
}

// Item of flat k-mer g, at or after item i (for the few threads whose k-mers
// span documents).
__device__ __noinline__ uint64_t item_at(const InsertArgs &a, uint64_t i, uint64_t g) {
    while (a.kcum[i + 1] <= g) ++i;
    return i;
}

template <int ETA, int KIND>
__global__ void __launch_bounds__(IB_THREADS, 4) k_insert_bin_scatter(InsertArgs a, BinnedInsert b, uint64_t f0,
                                                                      uint64_t f1) {
    constexpr uint32_t TK = IB_TILE_RECORDS / ETA;  // k-mers per tile
    constexpr int KPT = TK / IB_THREADS;            // consecutive k-mers per thread
    static_assert(KPT * IB_THREADS * ETA == IB_TILE_RECORDS, "tile of whole k-mer rounds");
    static_assert(2 * (KPT - 1) < 32 && KPT - 1 + 32 <= 48, "a thread's windows lie in 96 bits");
    extern __shared__ unsigned long long ib_smem[];
    unsigned long long *s_sorted = ib_smem;                                        // the tile in bin order
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(s_sorted + IB_TILE_RECORDS);    // IB_MAX_BINS each:
    uint32_t *s_base = s_cnt + IB_MAX_BINS;                                        // the tile's share of the bin
    uint32_t *s_pre = s_base + IB_MAX_BINS;                                        // the tile's records before it
    const uint64_t T = a.kcum[a.n];
    const uint64_t e1 = f1 < T ? f1 : T;
    if (f0 >= e1) return;  // the whole CTA
    uint64_t per = (e1 - f0 + gridDim.x - 1) / gridDim.x;
    per = (per + TK - 1) / TK * TK;
    const uint64_t c0 = f0 + (uint64_t)blockIdx.x * per;
    if (c0 >= e1) return;  // the whole CTA
    const uint64_t c1 = c0 + per < e1 ? c0 + per : e1;
    for (uint32_t i = threadIdx.x; i < b.nbins; i += IB_THREADS) s_cnt[i] = 0;
    __syncthreads();

    // document of this thread's first k-mer (largest i with kcum[i] <= g)
    const uint64_t g_first = c0 + threadIdx.x * KPT < c1 ? c0 + threadIdx.x * KPT : c1 - 1;
    uint64_t lo = 0, hi = a.n;
    while (hi - lo > 1) {
        const uint64_t mid = (lo + hi) >> 1;
        if (a.kcum[mid] <= g_first) lo = mid;
        else hi = mid;
    }
    const uint64_t item_first = lo;
    RecordSetter<KIND> set(a, threadIdx.x & 31);

    for (uint32_t jb = 0; jb < a.eta; jb += ETA) {
        uint64_t item = item_first, item_end = a.kcum[item + 1];
        for (uint64_t base = c0; base < c1; base += TK) {
            // 1. the thread's k-mers; its document only goes forward from tile
            //    to tile
            const uint64_t g0 = base + threadIdx.x * KPT;
            bool whole = false;  // all of one document
            uint32_t doc = NO_DOC, live = 0;
            uint32_t y[3];
            if (g0 < c1) {
                while (item_end <= g0) item_end = a.kcum[++item + 1];
                whole = g0 + KPT <= (item_end < c1 ? item_end : c1);
                if (whole) {
                    doc = a.doc_ids[item];
                    live = doc < a.K ? (1u << KPT) - 1 : 0u;
                    window96(a.packed, a.packed_bytes, a.offsets[item] + a.base_shift + (g0 - a.kcum[item]), y);
                }
            }
            // 2. the records' positions, ranked within their bins (two ranks to
            //    a register)
            uint32_t pos[KPT][ETA], rank[(KPT * ETA + 1) / 2];
#pragma unroll
            for (int j = 0; j < KPT; ++j) {
                uint64_t c = 0;
                if (whole) {
                    const uint32_t x0 = __funnelshift_r(y[0], y[1], 2 * j), x1 = __funnelshift_r(y[1], y[2], 2 * j);
                    c = canonical_from_window((uint64_t)x1 << 32 | x0, a.k);
                } else if (g0 + j < c1) {
                    const uint64_t i = item_at(a, item, g0 + j);
                    if (a.doc_ids[i] < a.K) {
                        const uint64_t t = a.offsets[i] + a.base_shift + (g0 + j - a.kcum[i]);
                        c = canonical_from_window(base_window(a.packed, a.packed_bytes, t), a.k);
                        live |= 1u << j;
                    }
                }
                const uint64_t km = mh_mix_key(c);
#pragma unroll
                for (int e = 0; e < ETA; ++e) {
                    uint32_t at = 0;
                    if (((live >> j) & 1u) && jb + e < a.eta) {
                        const uint64_t h = mh_first_word(km, a.seed32 + jb + e);
                        pos[j][e] = reduce_pos(h, a.m, a.m_inv);
                        at = atomicAdd(&s_cnt[pos[j][e] >> b.rshift], 1u);
                    }
                    const int x = j * ETA + e;
                    if (x & 1) rank[x / 2] |= at << 16;
                    else rank[x / 2] = at;
                }
            }
            __syncthreads();
            // 3. each bin's share of the global bin, one atomic per bin, and
            //    the tile's bin offsets
            for (uint32_t i = threadIdx.x; i < b.nbins; i += IB_THREADS) {
                const uint32_t n = s_cnt[i];
                s_base[i] = n ? atomicAdd(b.count + i, n) : 0u;
                s_pre[i] = n;
                s_cnt[i] = 0;
            }
            __syncthreads();
            const uint32_t total = ib_block_scan(s_pre, b.nbins);
            // 4. the tile in bin order
#pragma unroll
            for (int j = 0; j < KPT; ++j) {
                if (!((live >> j) & 1u)) continue;
                const uint32_t d = whole ? doc : a.doc_ids[item_at(a, item, g0 + j)];
#pragma unroll
                for (int e = 0; e < ETA; ++e) {
                    if (jb + e >= a.eta) break;
                    const int x = j * ETA + e;
                    s_sorted[s_pre[pos[j][e] >> b.rshift] + ((rank[x / 2] >> (16 * (x & 1))) & 0xffffu)] =
                        ((unsigned long long)pos[j][e] << IB_DOC_BITS) | d;
                }
            }
            __syncthreads();
            // 5. the records, or their bits when the bin is full
            for (uint32_t i0 = 0; i0 < total; i0 += IB_THREADS) {
                const uint32_t i = i0 + threadIdx.x;
                unsigned long long rec = 0;
                bool full = false;
                if (i < total) {
                    rec = s_sorted[i];
                    const uint32_t bin = record_group(rec) >> b.rshift;
                    const uint64_t at = (uint64_t)s_base[bin] + (i - s_pre[bin]);
                    full = at >= b.cap;
                    if (!full) b.buf[(uint64_t)bin * b.cap + at] = rec;
                }
                if (__any_sync(0xffffffffu, full)) set(record_group(rec), full ? record_doc(rec) : NO_DOC);
            }
            __syncthreads();  // the sorted tile is the next one's
        }
    }
}

// Apply pass: units of IB_UNIT records, claimed in bin order.  A CTA keeps
// IB_RING units of records under way into shared memory (their latency grows
// long beside the reductions) and one more claimed, while its warps set the
// records of the oldest: as in RecordSetter, neighbouring lanes take one
// record's words or repetitions, but each lane reads its record from the
// staged unit, so nothing is shuffled.  Bound by the L2 reductions: 2*10^9
// records of 16-byte groups take 10.5 ms in 16 MiB regions (12.9 in 32 MiB,
// 17.6 in 64 MiB, which each die's half of L2 no longer holds), against 22.1 ms
// with a thread per record and 14.6 ms with the warps' records shuffled.
// SPAT: the documents' patterns in shared memory (a gather of 16 patterns from
// L1 takes as long as the 32 reductions).
constexpr uint32_t IB_RING = 3;

// 16-byte copy to shared memory, read once: evict-first in L2.
__device__ __forceinline__ void copy_once(void *smem, const void *gmem, uint64_t policy) {
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(smem)),
                 "l"(gmem), "l"(policy)
                 : "memory");
}

constexpr size_t apply_smem(size_t pattern) { return (size_t)IB_RING * IB_UNIT * 8 + pattern; }

// SMALL: units of fewer records where the batch has less than one of IB_UNIT for
// every CTA; a thousand records in a warp wait for one another's latency (10^5
// k-mers on 64-byte groups: the whole insertion 102 us in full units, 61 so; the
// counts made by variables cost the medium build 2%, so it has its own template).
template <int KIND, bool SPAT, bool SMALL>
__global__ void __launch_bounds__(IB_THREADS) k_insert_bin_apply(InsertArgs a, BinnedInsert b) {
    extern __shared__ uint4 ib_apply_smem[];
    unsigned long long *ring = reinterpret_cast<unsigned long long *>(ib_apply_smem);  // IB_RING x IB_UNIT
    unsigned long long *s_pattern = ring + IB_RING * IB_UNIT;                          // SPAT: K x lanes
    __shared__ uint32_t s_pre[IB_MAX_BINS + 1];  // units before bin i
    __shared__ uint32_t s_unit[IB_RING + 1];     // claimed units
    __shared__ uint32_t s_have[IB_RING];         // records of the staged units
    // records per unit: IB_UNIT; SMALL: less when that leaves CTAs without one
    uint32_t unit = IB_UNIT;
    if constexpr (SMALL) {
        __shared__ uint32_t s_total;  // records of all bins (fewer than 2^32: see the launch)
        if (threadIdx.x == 0) s_total = 0;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < b.nbins; i += IB_THREADS) {
            const uint64_t n = b.count[i] < b.cap ? b.count[i] : b.cap;
            if (n) atomicAdd(&s_total, (uint32_t)n);
        }
        __syncthreads();
        while (unit > IB_UNIT_MIN && s_total < (uint64_t)gridDim.x * unit) unit /= 2;
    }
    // units per bin, then their exclusive prefix (warp 0: lane l sums bins
    // l*PER .. l*PER + PER - 1, a warp scan, then each lane writes its run)
    for (uint32_t i = threadIdx.x; i < b.nbins; i += IB_THREADS) {
        const uint64_t n = b.count[i] < b.cap ? b.count[i] : b.cap;
        s_pre[i] = (uint32_t)((n + unit - 1) / unit);
    }
    if (SPAT)
        for (uint32_t i = threadIdx.x; i < a.K * a.lanes; i += IB_THREADS) s_pattern[i] = __ldg(a.pattern + i);
    uint32_t *claim = b.count + IB_MAX_BINS;
    if (threadIdx.x == 0) {
        const uint32_t u = atomicAdd(claim, IB_RING + 1);
        for (uint32_t k = 0; k <= IB_RING; ++k) s_unit[k] = u + k;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        constexpr uint32_t PER = IB_MAX_BINS / 32;
        const uint32_t lane = threadIdx.x, i0 = lane * PER;
        uint32_t sum = 0;
        for (uint32_t i = i0; i < i0 + PER; ++i) sum += i < b.nbins ? s_pre[i] : 0u;
        uint32_t incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= (uint32_t)off) incl += o;
        }
        uint32_t run = incl - sum;
        for (uint32_t i = i0; i < i0 + PER && i < b.nbins; ++i) {
            const uint32_t u = s_pre[i];
            s_pre[i] = run;
            run += u;
        }
        if (lane == 31) s_pre[b.nbins] = incl;
    }
    __syncthreads();
    const uint32_t units = s_pre[b.nbins];
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    // starts the copy of claim j (one commit group, empty past the last unit)
    auto fetch = [&](uint32_t j) {
        const uint32_t u = s_unit[j % (IB_RING + 1)];
        if (u < units) {
            // the bin holding unit u: s_pre[lo] <= u < s_pre[lo + 1]
            uint32_t lo = 0, hi = b.nbins;
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if (s_pre[mid] <= u) lo = mid;
                else hi = mid;
            }
            const uint64_t n = b.count[lo] < b.cap ? b.count[lo] : b.cap;
            const uint64_t r0 = (uint64_t)(u - s_pre[lo]) * unit;
            const uint32_t have = n - r0 < unit ? (uint32_t)(n - r0) : unit;
            unsigned long long *to = ring + j % IB_RING * IB_UNIT;
            const unsigned long long *from = b.buf + (uint64_t)lo * b.cap + r0;
            // pairs of records (bins hold an even number of slots)
            for (uint32_t i = 2 * threadIdx.x; i < have; i += 2 * IB_THREADS) copy_once(to + i, from + i, policy);
            if (threadIdx.x == 0) s_have[j % IB_RING] = have;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (uint32_t j = 0; j + 1 < IB_RING; ++j) fetch(j);
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t per = 32 / a.lanes, sub = lane / a.lanes, part = lane - sub * a.lanes;
    const uint32_t share = (SMALL ? unit : IB_UNIT) / (IB_THREADS / 32);  // records of a unit per warp
    const uint32_t w0 = (threadIdx.x >> 5) * share;
    uint32_t next = 0;
    for (uint32_t j = 0;; ++j) {
        if (s_unit[j % (IB_RING + 1)] >= units) break;  // the whole CTA (claims increase)
        // (the unit whose stage this is was set before the last barrier)
        fetch(j + IB_RING - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(IB_RING - 1) : "memory");
        // claim j + IB_RING, made during the last unit, where claim j - 1 was
        if (threadIdx.x == 0 && j > 0) s_unit[(j + IB_RING) % (IB_RING + 1)] = next;
        __syncthreads();
        if (threadIdx.x == 0) next = atomicAdd(claim, 1u);
        const unsigned long long *rec = ring + j % IB_RING * IB_UNIT + w0;
        const uint32_t have = s_have[j % IB_RING];
        const uint32_t n = have > w0 ? (have - w0 < share ? have - w0 : share) : 0u;
        if (sub < per) {
#pragma unroll 4
            for (uint32_t i = sub; i < n; i += per) {
                const unsigned long long r = rec[i];
                const uint32_t p = record_group(r), d = record_doc(r);
                if (KIND == 0) {
                    for (uint32_t rep = part; rep < a.R; rep += a.lanes) {
                        const uint64_t bb =
                            (uint64_t)p * a.Gw * 32 + rep * a.B + __ldg(a.phi + (uint64_t)d * a.R + rep);
                        atomicOr(a.index + (bb >> 5), 1u << (bb & 31));
                    }
                } else if (KIND == 1) {
                    const unsigned long long bits =
                        SPAT ? s_pattern[d * a.lanes + part] : __ldg(a.pattern + (uint64_t)d * a.lanes + part);
                    atomicOr(reinterpret_cast<unsigned long long *>(a.index) + (uint64_t)p * a.lanes + part, bits);
                } else {
                    atomicOr(a.index + p, __ldg(reinterpret_cast<const uint32_t *>(a.pattern) + d));
                }
            }
        }
        __syncthreads();  // the stage and the claim are the next ones'
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// (most: what any launch of the kernel takes; the limit belongs to the kernel,
// so launches of several threads must not lower one another's)
template <typename KernelT>
int ib_blocks_per_sm(KernelT kernel, size_t smem, size_t most) {
    int n = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, IB_THREADS, smem) != cudaSuccess || n < 1)
        n = 1;
    return n;
}

// Blocks per resident block, as in the direct insertion (medium build: 21.8 ms
// with 1, 21.1 with 4, 20.7 with 16, 20.8 with 32).
constexpr int SCATTER_WAVES = 16;

template <int ETA, int KIND>
cudaError_t launch_scatter(const InsertArgs &a, const BinnedInsert &b, uint64_t f0, uint64_t f1, int sm_count,
                           cudaStream_t s) {
    const auto kernel = k_insert_bin_scatter<ETA, KIND>;
    const int occ = ib_blocks_per_sm(kernel, scatter_smem(), scatter_smem());
    uint64_t blocks = (uint64_t)sm_count * occ * SCATTER_WAVES;
    const uint64_t last = a.max_kmers && a.max_kmers < f1 ? a.max_kmers : f1;
    const uint64_t tiles = (last - f0 + IB_TILE_RECORDS / ETA - 1) / (IB_TILE_RECORDS / ETA);  // (f0 < max_kmers)
    if (blocks > tiles) blocks = tiles;
    kernel<<<(unsigned)blocks, IB_THREADS, scatter_smem(), s>>>(a, b, f0, f1);
    return cudaGetLastError();
}

// Patterns of up to this many bytes go to shared memory.
constexpr uint64_t IB_PATTERN_MAX = 32 * 1024;

template <int KIND, bool SPAT, bool SMALL>
cudaError_t launch_apply_t(const InsertArgs &a, const BinnedInsert &b, int sm_count, cudaStream_t s) {
    const auto kernel = k_insert_bin_apply<KIND, SPAT, SMALL>;
    const size_t smem = apply_smem(SPAT ? (size_t)a.K * a.lanes * 8 : 0);
    const int occ = ib_blocks_per_sm(kernel, smem, apply_smem(SPAT ? IB_PATTERN_MAX : 0));
    kernel<<<sm_count * occ, IB_THREADS, smem, s>>>(a, b);
    return cudaGetLastError();
}

template <int KIND, bool SPAT>
cudaError_t launch_apply(const InsertArgs &a, const BinnedInsert &b, int sm_count, cudaStream_t s) {
    // (five resident blocks an SM at most: 48 KB of shared memory each)
    const bool small = a.max_kmers && a.max_kmers < (uint64_t)sm_count * 5 * IB_UNIT / a.eta;
    return small ? launch_apply_t<KIND, SPAT, true>(a, b, sm_count, s) : launch_apply_t<KIND, SPAT, false>(a, b, sm_count, s);
}

template <int KIND>
cudaError_t launch_binned_k(const InsertArgs &a, const BinnedInsert &b, uint64_t f0, uint64_t f1, int sm_count,
                            cudaStream_t s) {
    cudaError_t e;
    if (a.eta == 1) e = launch_scatter<1, KIND>(a, b, f0, f1, sm_count, s);
    else if (a.eta == 2) e = launch_scatter<2, KIND>(a, b, f0, f1, sm_count, s);
    else e = launch_scatter<4, KIND>(a, b, f0, f1, sm_count, s);
    if (e != cudaSuccess) return e;
    if constexpr (KIND == 1)
        if ((uint64_t)a.K * a.lanes * 8 <= IB_PATTERN_MAX) return launch_apply<KIND, true>(a, b, sm_count, s);
    return launch_apply<KIND, false>(a, b, sm_count, s);
}

}  // namespace

uint32_t binned_insert_bins(uint64_t m, uint32_t group_bytes, uint32_t K, uint64_t region_bytes,
                            uint32_t *rshift) {
    if (m == 0 || group_bytes == 0 || m > (1ull << (64 - IB_DOC_BITS)) || K > (1u << IB_DOC_BITS)) return 0;
    uint32_t sh = 0;
    while (sh < 40 && ((uint64_t)group_bytes << (sh + 1)) <= region_bytes) ++sh;
    const uint64_t bins = (m + (1ull << sh) - 1) >> sh;
    if (bins > IB_MAX_BINS) return 0;
    *rshift = sh;
    return (uint32_t)bins;
}

cudaError_t launch_insert_binned(const InsertArgs &a, const BinnedInsert &b, uint64_t f0, uint64_t f1,
                                 int sm_count, cudaStream_t s) {
    if (a.lanes < 1 || a.lanes > 32) return cudaErrorInvalidValue;  // a turn holds at least one record
    switch (a.kind) {
        case 0: return launch_binned_k<0>(a, b, f0, f1, sm_count, s);
        case 1: return launch_binned_k<1>(a, b, f0, f1, sm_count, s);
        default: return launch_binned_k<2>(a, b, f0, f1, sm_count, s);
    }
}

}  // namespace rgpu
