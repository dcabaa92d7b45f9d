// stage_map.cuh -- sets of row or column indices as bitmaps in shared memory,
// for the global-memory bins while their staging area is free: a sorted list
// of distinct indices and the position of any index in it without a sort or a
// binary search.
#pragma once

#include "common.cuh"

namespace rsai {

// bits: one per index 0..n-1; pre: number of set bits before each word (at most
// the bins' |I| <= 32768, so 16 bits).  6 bytes per 32 indices: n = 1e6 takes
// 188 KB of the staging area.  Sorting the same candidates (a few thousand, in
// the workspace slab) took 66 to 91 passes over L2, and a lookup a chain of
// 10 to 12 dependent loads; the map takes two shared loads.
struct StageMap {
    uint32_t *bits = nullptr;
    uint16_t *pre = nullptr;
    int words = 0;

    static __host__ __device__ size_t bytes(int64_t n) { return (size_t)((n + 31) / 32) * 6 + 16; }

    __device__ StageMap(char *stage, int stage_bytes, int64_t n) {
        if (bytes(n) > (size_t)stage_bytes) return;  // too many indices: the caller sorts and searches
        words = (int)((n + 31) / 32);
        bits = reinterpret_cast<uint32_t *>(stage);
        pre = reinterpret_cast<uint16_t *>(bits + words);
    }
    __device__ __forceinline__ bool on() const { return bits != nullptr; }

    template <class Team> __device__ void clear(const Team &team) const {
        for (int i = team.rank(); i < words; i += Team::SIZE) bits[i] = 0u;
        team.sync();
    }
    __device__ __forceinline__ void mark(int32_t v) const { atomicOr(&bits[v >> 5], 1u << (v & 31)); }
    __device__ __forceinline__ void unmark(int32_t v) const { atomicAnd(&bits[v >> 5], ~(1u << (v & 31))); }
    // position of v among the marked indices, -1 if it is not marked
    __device__ __forceinline__ int find(int32_t v) const {
        const uint32_t b = bits[v >> 5], m = 1u << (v & 31);
        return (b & m) ? (int)pre[v >> 5] + __popc(b & (m - 1u)) : -1;
    }
    // After marking: forms the prefix counts and, if there are at most cap
    // marked indices, writes them to out in ascending order (out may be NULL).
    // Returns their number.  Synchronises the team before and after.
    template <class Team> __device__ int finish(const Team &team, int32_t *out, int cap) const {
        team.sync();
        const int per = (words + Team::SIZE - 1) / Team::SIZE;
        const int w0 = min(words, team.rank() * per), w1 = min(words, w0 + per);
        int cnt = 0;
        for (int i = w0; i < w1; ++i) cnt += __popc(bits[i]);
        int total;
        int at = team.scan(cnt, &total);
        if (total <= cap) {
            for (int i = w0; i < w1; ++i) {
                uint32_t b = bits[i];
                pre[i] = (uint16_t)at;
                if (out) {
                    for (; b; b &= b - 1u) out[at++] = i * 32 + __ffs(b) - 1;
                } else {
                    at += __popc(b);
                }
            }
        }
        team.sync();
        return total;
    }
};

}  // namespace rsai
