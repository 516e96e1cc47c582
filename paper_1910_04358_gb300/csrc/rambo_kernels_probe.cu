// rambo_kernels_probe.cu -- probe kernels of the batched query.
//
//   probe  (Algorithm 2's BFU membership tests, Section 3.3 / 3.3.1): every
//          k-mer of every query is canonicalised and hashed eta times; each
//          probe reads ONE position group -- the bits of all R*B BFUs at that
//          position -- so the per-BFU AND over eta probes and over all k-mers
//          of a query is a plain bitwise AND of groups.  The result per query
//          is its bucket mask: bit r*B+b set iff "Q in BFU(M[b,r])".
#include "rambo_query_common.cuh"

namespace rgpu {
namespace {

// ---------------------------------------------------------------------------
// probe: sequences.
//
// Lane roles.  A position group is read by LPG lanes, each loading an SW-word
// slice (16 bytes when the group is >= 16 bytes), so one warp instruction
// reads 32/LPG whole groups as runs of full 32-byte sectors (probe_range).
// The batch is cut into tiles of at most `tile` k-mers of one query, numbered
// by a prefix scan (kcum); every warp takes consecutive tiles, ANDs a tile's
// groups over its lanes and writes one mask: a plain store when the query is a
// single tile, else an atomicAnd into the mask set to ones.  Bound by the DRAM
// lines of the gathers (128 bytes each, whatever the group).  A warp that
// walked k-mers regardless of their query had every lane flush its own slice at
// each query's end, 128 atomics for a 32-byte group.
// FEW (probe_few_items: small tiles): a query's tiles are ANDed together in shared
// memory first, one atomicAnd for all of a warp's (one for every tile of 128
// k-mers doubles the time of a single sequence of 3*10^7 bases).  A template of
// its own: the state it keeps costs the other batches 2-5% on groups of 64 and
// 128 bytes, whose instances are short of registers.
struct TileShare {
    uint32_t tile;      // k-mers
    uint32_t per;       // tiles a warp takes, at most, unless the warps would not cover the batch
    uint32_t resident;  // warps that are resident together
};

// FEW: shares that every resident warp gets before they grow past one tile.
constexpr uint32_t FEW_ROUNDS = 4;

template <int SW, int LPG, int ETA, bool FEW>
__global__ void __launch_bounds__(PROBE_THREADS, LPG == 1 ? 2 : 3) k_probe_tiles(ProbeArgs a, TileShare sh) {
    __shared__ uint32_t run_smem[FEW ? PROBE_THREADS / 32 : 1][LPG * SW];  // a query's mask over the warp's tiles
    const int lane = threadIdx.x & 31;
    const uint32_t word0 = blockIdx.y * (LPG * SW) + (lane % LPG) * SW;
    const uint64_t tiles = a.kcum[a.n];
    const uint64_t warp = (uint64_t)blockIdx.x * (PROBE_THREADS / 32) + (threadIdx.x >> 5);
    const uint64_t nwarps = (uint64_t)gridDim.x * (PROBE_THREADS / 32);
    // (The launch knows only the bases that the batch's buffer spans: items may
    // overlap and have more tiles, or be a few places in it and have far fewer.)
    const uint64_t busy = tiles / (FEW ? FEW_ROUNDS * sh.resident : sh.resident), even = (tiles + nwarps - 1) / nwarps;
    uint64_t mine = sh.per < busy ? sh.per : busy;
    if (mine < even) mine = even;
    const uint64_t t0 = warp * mine;
    if (t0 >= tiles) return;
    const uint64_t t1 = t0 + mine < tiles ? t0 + mine : tiles;
    // (each lane that holds a mask, the first LPG, has its words to itself)
    if (FEW && LPG >= 8 && lane < LPG)
#pragma unroll
        for (int w = 0; w < SW; ++w) run_smem[threadIdx.x >> 5][lane * SW + w] = FULL;
    uint64_t q = find_query_warp(a.kcum, a.n, t0, lane);
    uint64_t first = a.kcum[q], next = a.kcum[q + 1];
    for (uint64_t t = t0; t < t1; ++t) {
        while (t >= next) {
            ++q;
            first = next;
            next = a.kcum[q + 1];
        }
        const uint64_t b0 = a.offsets[q], nk = a.ends[q] - b0 - a.k + 1;  // (a query with tiles has k-mers)
        const uint64_t k0 = (t - first) * sh.tile, k1 = k0 + sh.tile < nk ? k0 + sh.tile : nk;
        Slice<SW> s = probe_counted<SW, LPG, ETA, false, true, LPG == 4>(a, b0, k0, k1, lane, word0, nullptr);
        if (lane >= LPG) continue;
        if (next - first == 1) {
            uint32_t *p = a.acc + q * a.Gw + word0;
            if constexpr (SW == 4) *reinterpret_cast<uint4 *>(p) = make_uint4(s.w[0], s.w[1], s.w[2], s.w[3]);
            else
#pragma unroll
                for (int w = 0; w < SW; ++w) p[w] = s.w[w];
            continue;
        }
        if constexpr (FEW) {
            // (before a query's first tile the wide instances hold ones, the
            // others skip the words: the form that spills least)
            uint32_t *run = run_smem[threadIdx.x >> 5] + lane * SW;
            const bool ends = t + 1 == t1 || t + 1 == next;
            if (LPG >= 8 || (t != t0 && t != first))
#pragma unroll
                for (int w = 0; w < SW; ++w) s.w[w] &= run[w];
#pragma unroll
            for (int w = 0; w < SW; ++w) run[w] = LPG >= 8 && ends ? FULL : s.w[w];
            if (!ends) continue;
        }
        flush_slice<SW>(a.acc, q, a.Gw, word0, s);
    }
}

// ---------------------------------------------------------------------------
// probe: single k-mers of the widest groups (each k-mer is its own query; no
// cross-k-mer AND, so the bucket mask is stored directly).  Every other
// geometry is probed and answered in one launch by the answer kernels.
template <int SW, int LPG, int ETA>
__global__ void __launch_bounds__(PROBE_THREADS) k_probe_kmers(ProbeArgs a) {
    constexpr int RIF = 4;  // rounds whose loads are in flight together
    constexpr int NT = LPG >= RIF ? 1 : RIF / LPG;
    constexpr int KPR = 32 / LPG;
    constexpr int ROUNDS = NT * LPG;
    constexpr int STEP = 32 * NT;
    const int lane = threadIdx.x & 31;
    const int sub = lane / LPG;
    const uint32_t word0 = blockIdx.y * (LPG * SW) + (lane % LPG) * SW;

    const uint64_t T = a.n;
    uint64_t c0, c1;
    warp_range<STEP>(T, a.min_chunk, c0, c1);
    if (c0 >= T) return;
    const uint64_t kbits = kmask(a.k);

    for (uint32_t jb = 0; jb < a.eta; jb += ETA) {
        for (uint64_t base = c0; base < c1; base += STEP) {
            uint32_t pos[NT][ETA];
            bool val[NT];
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const uint64_t g = base + (uint64_t)t * 32 + lane;
                val[t] = g < c1;
                uint64_t c = 0;
                if (val[t]) {
                    uint64_t code = a.kmers[g];
                    if (code & ~kbits) {
                        if (jb == 0) atomicOr(a.err, ERR_KMER_CODE);
                        code &= kbits;
                    }
                    c = canonical_from_forward(code, a.k);
                }
                const uint64_t km = mh_mix_key(c);
#pragma unroll
                for (int e = 0; e < ETA; ++e) {
                    const uint32_t j = jb + e < a.eta ? jb + e : a.eta - 1;
                    pos[t][e] = reduce_pos(mh_first_word(km, a.seed32 + j), a.m, a.m_inv);
                }
            }
#pragma unroll
            for (int rg = 0; rg < ROUNDS; rg += RIF) {
                Slice<SW> v[RIF][ETA];
                bool vs[RIF];
#pragma unroll
                for (int rr = 0; rr < RIF; ++rr) {
                    const int rho = rg + rr;
                    const int t = rho / LPG;
                    const int src = (rho % LPG) * KPR + sub;
                    vs[rr] = __shfl_sync(FULL, (int)val[t], src) != 0;
#pragma unroll
                    for (int e = 0; e < ETA; ++e) {
                        const uint32_t p = __shfl_sync(FULL, pos[t][e], src);
                        if (vs[rr]) v[rr][e] = ld_slice<SW>(a.index + (uint64_t)p * a.Gw + word0);
                        else slice_ones(v[rr][e]);
                    }
                }
#pragma unroll
                for (int rr = 0; rr < RIF; ++rr) {
                    if (!vs[rr]) continue;
                    const int rho = rg + rr;
                    const uint64_t g = base + (uint64_t)(rho / LPG) * 32 + (rho % LPG) * KPR + sub;
                    Slice<SW> x = v[rr][0];
#pragma unroll
                    for (int e = 1; e < ETA; ++e) slice_and(x, v[rr][e]);
                    uint32_t *p = a.acc + g * a.Gw + word0;
                    if (jb == 0) {
#pragma unroll
                        for (int w = 0; w < SW; ++w) p[w] = x.w[w];
                    } else {
#pragma unroll
                        for (int w = 0; w < SW; ++w) atomicAnd(p + w, x.w[w]);
                    }
                }
            }
        }
    }
}

// K-mers a warp takes, about: small enough that many more blocks than fit are
// handed out as SMs get free.  One even share per resident warp waits for the
// SMs farthest from the memory: the 32 GiB batch takes 12.84 ms that way, 10.35
// with 4,096 k-mers a warp, 10.27 with 512 and 10.26 with 256; 20,000 short
// reads 170, 170, 155 and 148 us.
constexpr uint64_t SEQ_SHARE = 256;
// Warps that are resident on an SM.
constexpr uint32_t SEQ_RESIDENT = 24;
// Most blocks for every resident one, which leaves a warp 4,000 k-mers and more
// of a batch that has them: where a batch is a few places in its buffer, every
// further block finds nothing to do (500 ranges of 1,000 k-mers in 1.25 GB,
// 64-byte groups: 540 us with a block for every 8,192 bases of the buffer, 62
// like this).
constexpr uint64_t SEQ_WAVES = 16;
constexpr uint32_t SEQ_TILE = 128, SEQ_TILE_MAX = 1024;

// sm_count > 0: sized by the batch; sm_count < 0: -sm_count CTAs
template <int SW, int LPG, int ETA>
cudaError_t launch_seqs_t(const ProbeArgs &a, const Geometry &g, uint32_t tile, int sm_count, cudaStream_t s) {
    constexpr uint64_t WARPS = PROBE_THREADS / 32;
    uint64_t blocks = (uint64_t)-(int64_t)sm_count;
    TileShare sh{tile, 0, 1};
    const bool few = a.few != 0;
    if (sm_count > 0) {
        sh.resident = (uint32_t)sm_count * SEQ_RESIDENT;
        const uint64_t tiles = a.n + a.max_kmers / tile;  // at least as many as items that do not overlap have
        uint64_t share = few ? SEQ_TILE_MAX : SEQ_SHARE;
        if (share < a.min_chunk) share = a.min_chunk;
        uint64_t want = few ? share / SEQ_TILE : share * tiles / (a.max_kmers ? a.max_kmers : 1);
        const uint64_t most = tiles / (few ? FEW_ROUNDS * sh.resident : sh.resident);  // keep every warp busy first
        if (want > most) want = most;
        sh.per = want < 1 ? 1 : want > 1024 ? 1024 : (uint32_t)want;
        blocks = (tiles + WARPS * sh.per - 1) / (WARPS * sh.per);
        const uint64_t cap = sh.resident / WARPS * SEQ_WAVES;
        if (blocks > cap) blocks = cap;
    }
    const dim3 grid((unsigned)blocks, g.chunks);
    if (few) k_probe_tiles<SW, LPG, ETA, true><<<grid, PROBE_THREADS, 0, s>>>(a, sh);
    else k_probe_tiles<SW, LPG, ETA, false><<<grid, PROBE_THREADS, 0, s>>>(a, sh);
    return cudaGetLastError();
}

template <int SW, int LPG>
cudaError_t launch_seqs_eta(const ProbeArgs &a, const Geometry &g, uint32_t tile, int sm, cudaStream_t s) {
    switch (g.eta) {
        case 1: return launch_seqs_t<SW, LPG, 1>(a, g, tile, sm, s);
        case 2: return launch_seqs_t<SW, LPG, 2>(a, g, tile, sm, s);
        case 3: return launch_seqs_t<SW, LPG, 3>(a, g, tile, sm, s);
        default: return launch_seqs_t<SW, LPG, 4>(a, g, tile, sm, s);
    }
}

template <int ETA>
cudaError_t launch_kmers_t(const ProbeArgs &a, const Geometry &g, int sm_count, cudaStream_t s) {
    static int occ = blocks_per_sm(k_probe_kmers<4, 32, ETA>, PROBE_THREADS, 0);
    const dim3 grid(sm_count > 0 ? sm_count * occ : -sm_count, g.chunks);
    k_probe_kmers<4, 32, ETA><<<grid, PROBE_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

// Twice the resident warps: with more items, one tile each fills the rounds
// (10,000 of 1,000 k-mers, 128-byte groups: 446 us, 468 with small tiles; 8,000
// of them 394 and 397).  512 k-mers a warp: with fewer, tiles of an even share
// are small already.
bool probe_few_items(uint64_t n, uint64_t max_kmers, int sm_count) {
    const uint64_t warps = (uint64_t)sm_count * SEQ_RESIDENT;
    return n < 2 * warps && max_kmers >= 512 * warps;
}

// 1,024 (of 16 or more rounds of loads), fewer when that leaves warps without
// a tile.
uint32_t probe_tile_kmers(bool few, uint64_t max_kmers, int sm_count) {
    if (few) return SEQ_TILE;
    const uint64_t t = max_kmers / ((uint64_t)sm_count * SEQ_RESIDENT) / 64 * 64;
    return (uint32_t)(t < SEQ_TILE ? SEQ_TILE : t > SEQ_TILE_MAX ? SEQ_TILE_MAX : t);
}

cudaError_t launch_probe_seqs(const ProbeArgs &a, const Geometry &g, uint32_t tile, int sm_count, cudaStream_t s) {
    if (g.SW == 1) return launch_seqs_eta<1, 1>(a, g, tile, sm_count, s);
    if (g.SW == 2) return launch_seqs_eta<2, 1>(a, g, tile, sm_count, s);
    switch (g.LPG) {
        case 1: return launch_seqs_eta<4, 1>(a, g, tile, sm_count, s);
        case 2: return launch_seqs_eta<4, 2>(a, g, tile, sm_count, s);
        case 4: return launch_seqs_eta<4, 4>(a, g, tile, sm_count, s);
        case 8: return launch_seqs_eta<4, 8>(a, g, tile, sm_count, s);
        case 16: return launch_seqs_eta<4, 16>(a, g, tile, sm_count, s);
        case 32: return launch_seqs_eta<4, 32>(a, g, tile, sm_count, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_probe_kmers(const ProbeArgs &a, const Geometry &g, int sm_count, cudaStream_t s) {
    if (g.SW != 4 || g.LPG != 32) return cudaErrorInvalidValue;
    switch (g.eta) {
        case 1: return launch_kmers_t<1>(a, g, sm_count, s);
        case 2: return launch_kmers_t<2>(a, g, sm_count, s);
        default: return launch_kmers_t<4>(a, g, sm_count, s);
    }
}

}  // namespace rgpu
