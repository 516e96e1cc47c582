// rambo_insert_common.cuh -- setting the bits of probe records, shared by the
// direct and the region-binned insertion (device code).
#pragma once

#include "rambo_internal.cuh"

namespace rgpu {
namespace {

constexpr uint32_t NO_DOC = 0xffffffffu;

// A record is a position group p and a document d; setting it ORs bit
// r*B + phi_r(d) of the group for every r.  The lanes of a warp share the
// records: `lanes` consecutive lanes take one record, each one word (KIND 1,
// 2) or one repetition (KIND 0, more than 32 of them in turns) of it, so that
// a record's atomics leave in one instruction and reach L2 as one request per
// line.  One lane per record with its atomics in sequence sends a request for
// each: on 64-byte groups with R = 5 that ran at 8.6 G records/s over 4 GiB
// and 43.8 G/s in L2, against 22.7 and 105.5 this way (256-byte groups, R =
// 6: 6.6 and 34.7 against 15.3 and 40.6; 16-byte groups: 20.0 and 104 against
// 22.9 and 193).
//   KIND 0  repetitions, 32-bit words, buckets from phi
//   KIND 1  the 64-bit words of the group, from the documents' patterns
//           (at most R / 2 of them, so that nearly all have a bit, and at
//           most 32)
//   KIND 2  the one 32-bit word of a 4-byte group, from its pattern
template <int KIND>
struct RecordSetter {
    const InsertArgs &a;
    uint32_t sub, mine, per;  // this lane's record of a turn, its part of it, records a turn
    uint32_t cur_d;           // document whose part is at hand
    uint64_t bits;            // KIND 0: bit of the group; else the word's bits

    __device__ __forceinline__ RecordSetter(const InsertArgs &args, int lane) : a(args), cur_d(NO_DOC), bits(0) {
        per = 32 / a.lanes;
        sub = (uint32_t)lane / a.lanes;
        mine = (uint32_t)lane - sub * a.lanes;
    }

    __device__ __forceinline__ void fetch(uint32_t d, uint32_t part) {
        if (KIND == 0) bits = part * a.B + __ldg(a.phi + (uint64_t)d * a.R + part);
        else if (KIND == 1) bits = __ldg(a.pattern + (uint64_t)d * a.lanes + part);
        else bits = __ldg(reinterpret_cast<const uint32_t *>(a.pattern) + d);
    }

    __device__ __forceinline__ void set(uint32_t p) const {
        if (KIND == 0) {
            const uint64_t bb = (uint64_t)p * a.Gw * 32 + bits;
            atomicOr(a.index + (bb >> 5), 1u << (bb & 31));
        } else if (KIND == 1) {
            if (bits)
                atomicOr(reinterpret_cast<unsigned long long *>(a.index) + (uint64_t)p * a.lanes + mine,
                         (unsigned long long)bits);
        } else {
            atomicOr(a.index + p, (uint32_t)bits);
        }
    }

    // Sets the warp's 32 records (this lane's: group p, document d, or NO_DOC
    // for none).  Every lane of the warp calls it.
    __device__ __forceinline__ void operator()(uint32_t p, uint32_t d) {
        if (!__any_sync(0xffffffffu, d != NO_DOC)) return;
        for (uint32_t i = 0; i < 32; i += per) {
            const uint32_t src = i + sub;
            const uint32_t pp = __shfl_sync(0xffffffffu, p, src & 31);
            const uint32_t dd = __shfl_sync(0xffffffffu, d, src & 31);
            if (sub >= per || src > 31 || dd == NO_DOC) continue;
            if (KIND == 0 && a.R > 32) {
                for (uint32_t r = mine; r < a.R; r += a.lanes) {
                    fetch(dd, r);
                    set(pp);
                }
            } else {
                if (dd != cur_d) {
                    fetch(dd, mine);
                    cur_d = dd;
                }
                set(pp);
            }
        }
    }
};

}  // namespace
}  // namespace rgpu
