// rambo_kernels_answers.cu -- answers from bucket masks, 32 queries at a time
// (Algorithm 2's union and intersection), and the single-k-mer query that
// probes and answers in the same launch.
//
// Every repetition partitions the documents, so document d is in a query's
// answer iff the query's bucket mask has bit r*B + phi_r(d) set for every r
// (Algorithm 2: d is in the union of repetition r's passing buckets iff its
// own bucket passes).  A warp takes a group of 32 queries and turns their
// masks on their side: word s of its table M holds bit s of all 32 masks.
// A lane that owns document d then answers it for the 32 queries at once,
// with R shared-memory reads and R - 1 ANDs, and a 32 x 32 bit transpose
// across the warp gives every lane one word of its query's answer.
//
// What bounds it: the shared-memory pipe (per 32 documents x 32 queries: R
// table reads, R/2 reads of the documents' slots, 4 shuffles of the
// transpose, 3 accesses to stage and store the words), then the stores of the
// answers.  Each query's share is about 1 / 30 of the table reads of an
// expansion row by row: 10^6 k-mers over 1,000 documents (1 GiB index) take
// 87 us, probe included, against 206 us for a probe launch and a nibble-table
// expansion; 10^5 over 10,000 documents 111 us against 1,850 us (byte table);
// the masks of 20,000 sequences over 500 documents 4 against 30 us.
// Three blocks an SM: with four or five (fewer registers each) the 10^6
// k-mers take 89 and 97 us, and 10^5 over 10,000 documents 112 and 115 us.
#include "rambo_query_common.cuh"

namespace rgpu {
namespace {

constexpr int ANS_THREADS = 256;
constexpr int ANS_WARPS = ANS_THREADS / 32;
constexpr uint32_t ANS_QUADS = 8;                   // 4-word quads staged before they are stored
constexpr uint32_t ANS_PITCH = 4 * ANS_QUADS + 4;   // words: 16-byte accesses of 8 rows hit all banks
constexpr uint32_t ANS_STAGE = 32 * ANS_PITCH;      // words per warp
// Units per worker a batch is split for.  A unit pays for its own table, so
// more units cost more: 10^5 k-mers over 10,000 documents take 119 us at 1 or
// 2 units a worker, 111 us at 4, and (before the tables' rows came coalesced
// through the stage) 135, 142, 165 and 235 us at 1, 2, 4 and 8.
constexpr uint64_t ANS_UNITS = 4;
// Most slots of M that 16-bit byte offsets address, the empty slot included.
constexpr uint32_t ANS_MAX_SLOTS = 16384;
// Tables up to this size are kept one per warp (three blocks an SM still
// fit); larger ones are shared by the block's warps, which then wait for one
// another around each group.
constexpr uint32_t ANS_WARP_TABLE_MAX = 2112;       // words

struct AnswerArgs {
    ProbeArgs p;             // PROBE: index, hashing and the k-mers
    const uint32_t *acc;     // otherwise: n x Gw bucket masks
    uint64_t n;
    uint32_t Gw, R, RB, W;
    const uint32_t *slots;   // answer_slot_words: byte offsets of the documents' slots in M
    uint32_t *out;           // n x W
    uint32_t quads;          // ceil(W / 4)
    uint32_t quads_per_unit, units_per_group;
    uint32_t m_words;        // words of one table M (a multiple of 4)
};

// Lane i holds row i of a 32 x 32 bit matrix, four matrices at once; on
// return lane i holds column i.  Butterflies over lane distance 16 and 8
// exchange whole bytes: two words share one shuffle, packed and unpacked by
// byte permutes.  Distances 4, 2, 1 rotate and merge.
struct Transpose {
    uint32_t selp16, sela16, selb16, selp8, sela8, selb8;
    uint32_t rot[3], keep[3];

    __device__ __forceinline__ explicit Transpose(int lane) {
        // a low lane (bit clear) keeps the low bytes of each pair and sends
        // the high ones; a high lane the other way round
        const bool h16 = lane & 16, h8 = lane & 8;
        selp16 = h16 ? 0x5410 : 0x7632;  // sent: A's half in the low, B's in the high half
        sela16 = h16 ? 0x3254 : 0x5410;  // A' from A (0-3) and the received word (4-7)
        selb16 = h16 ? 0x3276 : 0x7610;
        selp8 = h8 ? 0x6420 : 0x7531;    // sent: A's two bytes, then B's two
        sela8 = h8 ? 0x3514 : 0x5240;
        selb8 = h8 ? 0x3716 : 0x7260;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int s = 4 >> i;
            const uint32_t m = s == 4 ? 0x0f0f0f0fu : s == 2 ? 0x33333333u : 0x55555555u;
            rot[i] = (lane & s) ? 32 - s : s;
            keep[i] = (lane & s) ? ~m : m;
        }
    }
    __device__ __forceinline__ static void bytes(uint32_t &a, uint32_t &b, int dist, uint32_t sp, uint32_t sa,
                                                 uint32_t sb) {
        const uint32_t q = __shfl_xor_sync(FULL, __byte_perm(a, b, sp), dist);
        a = __byte_perm(a, q, sa);
        b = __byte_perm(b, q, sb);
    }
    __device__ __forceinline__ void operator()(uint32_t (&v)[4]) const {
        bytes(v[0], v[1], 16, selp16, sela16, selb16);
        bytes(v[2], v[3], 16, selp16, sela16, selb16);
        bytes(v[0], v[1], 8, selp8, sela8, selb8);
        bytes(v[2], v[3], 8, selp8, sela8, selb8);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t y = __shfl_xor_sync(FULL, v[j], 4 >> i);
                const uint32_t z = __funnelshift_l(y, y, rot[i]);
                v[j] = (v[j] & keep[i]) | (z & ~keep[i]);
            }
    }
};

// Probe positions of a group's k-mers (lane = k-mer), seeds jb .. jb+ETA-1
// (past the last seed, the last one again).
template <int ETA>
__device__ __forceinline__ void kmer_rows(const AnswerArgs &a, uint64_t km, uint32_t jb, uint32_t (&row)[ETA]) {
#pragma unroll
    for (int e = 0; e < ETA; ++e) {
        const uint32_t j = jb + e < a.p.eta ? jb + e : a.p.eta - 1;
        row[e] = reduce_pos(mh_first_word(km, a.p.seed32 + j), a.p.m, a.p.m_inv);
    }
}

__device__ __forceinline__ uint64_t kmer_key(const AnswerArgs &a, uint64_t q) {
    const uint64_t kbits = kmask(a.p.k);
    uint64_t code = __ldg(reinterpret_cast<const unsigned long long *>(a.p.kmers) + q);
    if (code & ~kbits) {
        atomicOr(a.p.err, ERR_KMER_CODE);
        code &= kbits;
    }
    return mh_mix_key(canonical_from_forward(code, a.p.k));
}

// M of one group of 32 queries from rows of Gw words at base + row * Gw, the
// AND of ETA rows per query (lane = query, `row` its row numbers, live: the
// query exists).  Rows of 16 bytes and more come through the warp's stage:
// eight consecutive lanes copy 16-byte pieces of one query's rows, so that a
// row's pieces share their lines' requests.  A round covers 8 / ETA pieces of
// every row, rounds w0, w0 + step, ..; `first` starts M, else it is ANDed.
template <int ETA>
__device__ __forceinline__ void table_from_rows(const AnswerArgs &a, const uint32_t *base, const uint64_t (&row)[ETA],
                                                bool live, bool first, uint32_t *M, uint32_t *stage, uint32_t w0,
                                                uint32_t step, int lane, const Transpose &tr) {
    auto put = [&](uint32_t wq, uint32_t (&v)[4]) {
        tr(v);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t *m = M + (4 * wq + c) * 32 + lane;
            *m = first ? v[c] : *m & v[c];
        }
    };
    if ((a.Gw & 3) != 0) {  // groups of 4 or 8 bytes: one quad, read in place
        if (w0) return;
        uint32_t v[4] = {live ? FULL : 0u, live ? FULL : 0u, 0u, 0u};
        if (live) {
#pragma unroll
            for (int e = 0; e < ETA; ++e) {
                const uint32_t *p = base + row[e] * a.Gw;
                if (a.Gw == 2) {
                    const Slice<2> x = ld_slice<2>(p);
                    v[0] &= x.w[0];
                    v[1] &= x.w[1];
                } else {
                    v[0] &= ld_slice<1>(p).w[0];
                }
            }
        }
        put(0, v);
        return;
    }
    constexpr uint32_t QR = 8 / ETA;  // pieces of each row per round
    const uint32_t nq = a.Gw / 4;
    const uint32_t alive = __ballot_sync(FULL, live);
    const int piece = lane & 7, mine = piece / (int)QR;
    for (uint32_t wb = w0 * QR; wb < nq; wb += step * QR) {
        const uint32_t wq = wb + piece % QR;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int q = 4 * i + (lane >> 3);
            uint64_t r = __shfl_sync(FULL, row[0], q);
#pragma unroll
            for (int e = 1; e < ETA; ++e) {
                const uint64_t x = __shfl_sync(FULL, row[e], q);
                if (mine == e) r = x;
            }
            if (wq < nq && ((alive >> q) & 1u))
                cp_async16(reinterpret_cast<uint4 *>(stage + q * ANS_PITCH + 4 * piece), base + r * a.Gw + 4 * wq);
        }
        cp_async_wait_all();
        __syncwarp();
#pragma unroll
        for (uint32_t j = 0; j < QR; ++j) {
            if (wb + j >= nq) break;
            uint32_t v[4] = {0u, 0u, 0u, 0u};
            if (live) {
                const uint4 *s = reinterpret_cast<const uint4 *>(stage + lane * ANS_PITCH) + j;
                uint4 x = s[0];
#pragma unroll
                for (int e = 1; e < ETA; ++e) {
                    const uint4 y = s[e * QR];
                    x.x &= y.x; x.y &= y.y; x.z &= y.z; x.w &= y.w;
                }
                v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
            }
            put(wb + j, v);
        }
        __syncwarp();  // the stage is the next round's
    }
}

// Slot words of one document block: RT repetitions at compile time, or R (0: up
// to 16; -1: more).
template <int RT>
__device__ __forceinline__ uint32_t answer_word(const AnswerArgs &a, const char *M, uint32_t block, int lane) {
    auto at = [&](uint32_t off) { return *reinterpret_cast<const uint32_t *>(M + off); };
    if constexpr (RT > 0) {
        constexpr int RP = (RT + 1) / 2;
        const uint32_t *s = a.slots + (uint64_t)block * (RP * 32) + lane;
        uint32_t x[RP];
#pragma unroll
        for (int p = 0; p < RP; ++p) x[p] = __ldg(s + 32 * p);
        uint32_t v = FULL;
#pragma unroll
        for (int p = 0; p < RP; ++p) {
            v &= at(x[p] & 0xffffu);
            if (2 * p + 1 < RT) v &= at(x[p] >> 16);
        }
        return v;
    } else if constexpr (RT == 0) {
        const uint32_t rp = (a.R + 1) / 2;
        const uint32_t *s = a.slots + (uint64_t)block * (rp * 32) + lane;
        uint32_t v = FULL;
        for (uint32_t p = 0; p < rp; ++p) {
            const uint32_t x = __ldg(s + 32 * p);
            v &= at(x & 0xffffu);
            if (2 * p + 1 < a.R) v &= at(x >> 16);
        }
        return v;
    } else {
        // many repetitions: four pairs' slots at a time, and no more of them once
        // no query has any of these documents (R = 128, 5,000 documents, 20,000
        // random k-mers: 47 us, 240 one pair after the other to the end; with R =
        // 7..9 it costs 5-10%)
        const uint32_t rp = (a.R + 1) / 2;
        const uint32_t *s = a.slots + (uint64_t)block * (rp * 32) + lane;
        uint32_t v = FULL;
        for (uint32_t p0 = 0; p0 < rp; p0 += 4) {
            uint32_t x[4];
#pragma unroll
            for (uint32_t i = 0; i < 4; ++i) x[i] = p0 + i < rp ? __ldg(s + 32 * (p0 + i)) : 0u;
#pragma unroll
            for (uint32_t i = 0; i < 4; ++i) {
                if (p0 + i >= rp) break;
                v &= at(x[i] & 0xffffu);
                if (2 * (p0 + i) + 1 < a.R) v &= at(x[i] >> 16);
            }
            if (!__any_sync(FULL, v)) break;
        }
        return v;
    }
}

// The staged words [w0, w0 + nw) of the group's queries, 32 rows of ANS_PITCH
// words, to their answer rows.  Full tiles go row by row (or four rows of
// 16-byte accesses at a time, when the rows are aligned) at fixed strides.
// Others go in the order of the rows' words, so that consecutive lanes write
// consecutive words (division of an index below 1024 by nw <= 32 by a 16-bit
// reciprocal, exact there).
__device__ __forceinline__ void store_words(const AnswerArgs &a, const uint32_t *stage, uint64_t q0, uint32_t w0,
                                            uint32_t nw, bool vec, int lane) {
    const uint32_t rows = a.n - q0 < 32 ? (uint32_t)(a.n - q0) : 32u;
    uint32_t *out = a.out + q0 * a.W + w0;
    if (rows == 32 && nw == 4 * ANS_QUADS) {
        if (vec) {
            const uint32_t *from = stage + (lane >> 3) * ANS_PITCH + 4 * (lane & 7);
            uint32_t *to = out + (uint64_t)(lane >> 3) * a.W + 4 * (lane & 7);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<uint4 *>(to + (uint64_t)(4 * i) * a.W) =
                    *reinterpret_cast<const uint4 *>(from + 4 * i * ANS_PITCH);
        } else {
            uint32_t *to = out + lane;
#pragma unroll
            for (int i = 0; i < 32; ++i, to += a.W) *to = stage[i * ANS_PITCH + lane];
        }
    } else if (vec) {
        const uint32_t nv = nw / 4;  // W is a multiple of 4, so nw is too
        const uint32_t inv = (65536 + nv - 1) / nv;
        for (uint32_t i = lane; i < rows * nv; i += 32) {
            const uint32_t row = (i * inv) >> 16, c = i - row * nv;
            *reinterpret_cast<uint4 *>(out + (uint64_t)row * a.W + 4 * c) =
                *reinterpret_cast<const uint4 *>(stage + row * ANS_PITCH + 4 * c);
        }
    } else {
        const uint32_t inv = (65536 + nw - 1) / nw;
        for (uint32_t i = lane; i < rows * nw; i += 32) {
            const uint32_t row = (i * inv) >> 16, c = i - row * nw;
            out[(uint64_t)row * a.W + c] = stage[row * ANS_PITCH + c];
        }
    }
}

// One unit = (group of 32 queries, range of 128-document quads).  SHARED: a
// block takes a unit, its warps share the table and stride over the range;
// else every warp takes its own units.  ETA 0: masks from memory.
template <int RT, int ETA, bool SHARED>
__global__ void __launch_bounds__(ANS_THREADS, 3) k_answers(AnswerArgs a) {
    extern __shared__ uint4 ans_smem[];
    const int lane = threadIdx.x & 31;
    const int wib = __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0);  // the same in every lane: a uniform register
    uint32_t *smem = reinterpret_cast<uint32_t *>(ans_smem);
    uint32_t *stage = smem + wib * ANS_STAGE;
    uint32_t *M = smem + ANS_WARPS * ANS_STAGE + (SHARED ? 0 : wib * a.m_words);
    const Transpose tr(lane);
    const bool vec = (a.W & 3) == 0 && (reinterpret_cast<uintptr_t>(a.out) & 15) == 0;
    const uint64_t units = (a.n + 31) / 32 * a.units_per_group;
    const uint64_t first = SHARED ? blockIdx.x : (uint64_t)blockIdx.x * ANS_WARPS + wib;
    const uint64_t step = SHARED ? gridDim.x : (uint64_t)gridDim.x * ANS_WARPS;
    for (uint64_t u = first; u < units; u += step) {
        const uint64_t g = u / a.units_per_group;
        const uint64_t q0 = g * 32;
        const uint32_t b0 = (uint32_t)(u - g * a.units_per_group) * a.quads_per_unit;
        const uint32_t b1 = b0 + a.quads_per_unit < a.quads ? b0 + a.quads_per_unit : a.quads;
        const uint32_t w0 = SHARED ? wib : 0, wstep = SHARED ? ANS_WARPS : 1;
        const bool live = q0 + lane < a.n;
        if constexpr (ETA > 0) {
            const uint64_t km = live ? kmer_key(a, q0 + lane) : 0;
            for (uint32_t jb = 0; jb < a.p.eta; jb += ETA) {
                uint32_t pos[ETA];
                uint64_t row[ETA];
                kmer_rows<ETA>(a, km, jb, pos);
#pragma unroll
                for (int e = 0; e < ETA; ++e) row[e] = pos[e];
                table_from_rows<ETA>(a, a.p.index, row, live, jb == 0, M, stage, w0, wstep, lane, tr);
            }
        } else {
            const uint64_t row[1] = {q0 + lane};
            table_from_rows<1>(a, a.acc, row, live, true, M, stage, w0, wstep, lane, tr);
        }
        if (SHARED) __syncthreads();
        else __syncwarp();
        if ((!SHARED || wib == 0) && lane == 0) M[a.RB] = 0;  // the slot of documents not inserted
        if (SHARED) __syncthreads();
        else __syncwarp();
        for (uint32_t s = b0 + (SHARED ? wib * ANS_QUADS : 0u); s < b1; s += SHARED ? ANS_WARPS * ANS_QUADS : ANS_QUADS) {
            const uint32_t nq = b1 - s < ANS_QUADS ? b1 - s : ANS_QUADS;
            for (uint32_t t = 0; t < nq; ++t) {
                uint32_t v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    v[j] = answer_word<RT>(a, reinterpret_cast<const char *>(M), 4 * (s + t) + j, lane);
                tr(v);
                *reinterpret_cast<uint4 *>(stage + lane * ANS_PITCH + 4 * t) = make_uint4(v[0], v[1], v[2], v[3]);
            }
            __syncwarp();
            store_words(a, stage, q0, 4 * s, a.W - 4 * s < 4 * nq ? a.W - 4 * s : 4 * nq, vec, lane);
            __syncwarp();
        }
        if (SHARED) __syncthreads();
    }
}

template <int RT, int ETA, bool SHARED>
cudaError_t launch_answers_t(AnswerArgs &a, int max_blocks, int sm_count, cudaStream_t s) {
    const size_t smem = ((size_t)ANS_WARPS * ANS_STAGE + (size_t)a.m_words * (SHARED ? 1 : ANS_WARPS)) * 4;
    // (the limit belongs to the kernel, not to the launch: always the most that
    // any geometry takes, so that launches of several threads don't lower one
    // another's)
    constexpr size_t limit = ((size_t)ANS_WARPS * ANS_STAGE + (SHARED ? ANS_MAX_SLOTS : ANS_WARPS * ANS_WARP_TABLE_MAX)) * 4;
    if (smem > limit) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k_answers<RT, ETA, SHARED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)limit);
    if (e != cudaSuccess) return e;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_answers<RT, ETA, SHARED>, ANS_THREADS, smem);
    if (e != cudaSuccess) return e;
    uint64_t cap = (uint64_t)(occ > 0 ? occ : 1) * (uint64_t)sm_count;
    if (cap > (uint64_t)max_blocks) cap = (uint64_t)max_blocks;
    // few queries: split each group's documents so that every warp has work;
    // up to ANS_UNITS units a worker while a unit keeps 32 answer words, so
    // that the last round of units leaves few warps idle
    const uint64_t groups = (a.n + 31) / 32;
    const uint64_t workers = cap * (SHARED ? 1 : ANS_WARPS);
    uint64_t per_group = (workers + groups - 1) / groups;
    const uint64_t fine = (ANS_UNITS * workers + groups - 1) / groups, most = (a.quads + ANS_QUADS - 1) / ANS_QUADS;
    const uint64_t want = fine < most ? fine : most;
    if (per_group < want) per_group = want;
    uint64_t per = (a.quads + per_group - 1) / per_group;
    if (SHARED) per = (per + ANS_WARPS * ANS_QUADS - 1) / (ANS_WARPS * ANS_QUADS) * (ANS_WARPS * ANS_QUADS);
    else if (per > ANS_QUADS) per = (per + ANS_QUADS - 1) / ANS_QUADS * ANS_QUADS;
    a.quads_per_unit = (uint32_t)per;
    a.units_per_group = (uint32_t)((a.quads + per - 1) / per);
    const uint64_t units = groups * a.units_per_group;
    uint64_t blocks = SHARED ? units : (units + ANS_WARPS - 1) / ANS_WARPS;
    if (blocks > cap) blocks = cap;
    k_answers<RT, ETA, SHARED><<<(unsigned)blocks, ANS_THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

template <int RT, int ETA>
cudaError_t launch_answers_s(AnswerArgs &a, int max_blocks, int sm_count, cudaStream_t s) {
    return a.m_words <= ANS_WARP_TABLE_MAX ? launch_answers_t<RT, ETA, false>(a, max_blocks, sm_count, s)
                                           : launch_answers_t<RT, ETA, true>(a, max_blocks, sm_count, s);
}

template <int ETA>
cudaError_t launch_answers_r(AnswerArgs &a, int max_blocks, int sm_count, cudaStream_t s) {
    switch (a.R) {
        case 2: return launch_answers_s<2, ETA>(a, max_blocks, sm_count, s);
        case 3: return launch_answers_s<3, ETA>(a, max_blocks, sm_count, s);
        case 4: return launch_answers_s<4, ETA>(a, max_blocks, sm_count, s);
        case 5: return launch_answers_s<5, ETA>(a, max_blocks, sm_count, s);
        case 6: return launch_answers_s<6, ETA>(a, max_blocks, sm_count, s);
        default:
            return a.R <= 16 ? launch_answers_s<0, ETA>(a, max_blocks, sm_count, s)
                             : launch_answers_s<-1, ETA>(a, max_blocks, sm_count, s);
    }
}

AnswerArgs answer_args(const Geometry &g, uint64_t n, const uint32_t *slots, uint32_t *out) {
    AnswerArgs a{};
    a.n = n;
    a.Gw = g.Gw;
    a.R = g.R;
    a.RB = g.gbits;
    a.W = g.W;
    a.slots = slots;
    a.out = out;
    a.quads = (g.W + 3) / 4;
    const uint32_t words = 32 * ((g.Gw + 3) / 4 * 4);
    a.m_words = (words > g.gbits ? words : g.gbits + 1) + 3 & ~3u;
    return a;
}

// Every slot to the empty one (no document inserted).
__global__ void k_slots_fill(uint32_t *slots, uint64_t words, uint32_t pair) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += (uint64_t)gridDim.x * blockDim.x)
        slots[i] = pair;
}

// The slots of every inserted document (bit d of its bucket's bitmap set).
__global__ void k_slots_rebuild(uint16_t *slots, const uint32_t *docbits, const uint32_t *phi, uint32_t K, uint32_t R,
                                uint32_t B, uint32_t W) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (uint64_t)K * R) return;
    const uint32_t d = (uint32_t)(i / R), r = (uint32_t)(i % R);
    const uint32_t b = phi[i];
    if ((docbits[((uint64_t)r * B + b) * W + (d >> 5)] >> (d & 31)) & 1u)
        slots[answer_slot_index(d, r, R)] = (uint16_t)(4 * (r * B + b));
}

}  // namespace

uint64_t answer_slot_words(const Geometry &g) {
    if (g.gbits + 1 > ANS_MAX_SLOTS) return 0;
    return (uint64_t)((g.W + 3) / 4 * 4) * 32 * ((g.R + 1) / 2);
}

cudaError_t launch_slots(const Geometry &g, uint32_t *slots, const uint32_t *docbits, const uint32_t *phi,
                         int sm_count, cudaStream_t s) {
    const uint32_t empty = 4 * g.gbits;
    k_slots_fill<<<sm_count * 4, 256, 0, s>>>(slots, answer_slot_words(g), empty | (empty << 16));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !docbits) return e;
    const uint64_t n = (uint64_t)g.K * g.R;
    k_slots_rebuild<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(reinterpret_cast<uint16_t *>(slots), docbits, phi, g.K,
                                                                g.R, g.B, g.W);
    return cudaGetLastError();
}

cudaError_t launch_answers(const Geometry &g, const uint32_t *acc, uint64_t n, const uint32_t *slots, uint32_t *out,
                           int max_blocks, int sm_count, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    AnswerArgs a = answer_args(g, n, slots, out);
    a.acc = acc;
    return launch_answers_r<0>(a, max_blocks, sm_count, s);
}

cudaError_t launch_kmer_answers(const ProbeArgs &p, const Geometry &g, const uint32_t *slots, uint32_t *out,
                                int max_blocks, int sm_count, cudaStream_t s) {
    if (p.n == 0) return cudaSuccess;
    AnswerArgs a = answer_args(g, p.n, slots, out);
    a.p = p;
    switch (g.eta) {
        case 1: return launch_answers_r<1>(a, max_blocks, sm_count, s);
        case 2: return launch_answers_r<2>(a, max_blocks, sm_count, s);
        default: return launch_answers_r<4>(a, max_blocks, sm_count, s);
    }
}

}  // namespace rgpu
