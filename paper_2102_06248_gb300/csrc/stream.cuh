// stream.cuh -- matrix-vector products of the persistent solvers, with the
// matrix streamed through shared memory by bulk copies.
//
// What bounds a sparse product here is memory latency: a thread that loads a
// column index, then gathers the vector entry it names, then multiplies has
// its stream idle while it waits for the gather.  With 32 warps an SM that
// left DRAM at about half its rate.  So the stream is taken out of the threads'
// hands: the matrix is stored as a sequence of records of kCols SELL columns
// (32 rows each), every warp owns a contiguous run of slices, hence a
// contiguous run of records, and one lane keeps a ring of bulk copies
// (cp.async.bulk into shared memory, completion on an mbarrier) in flight ahead
// of the warp, across slice ends, grid barriers and iterations.  The warp's
// own loads are then the gathers only, kCols of them at a time.
//
// A record holds kCols x 32 values and the columns.  NARROW columns are one
// byte an entry and one 32-bit base per SELL column (column = base + lane +
// byte): 5.1 bytes a nonzero in FP32 instead of 8, 9.1 instead of 12 in FP64.
// The slots of a slice are assigned so that its lanes' columns in a slot lie
// within a byte of each other (mesh.cpp); a matrix where that does not work out
// has WIDE records with 32-bit columns.
//   values   FP32: 2 planes [32 lanes][4], FP64: 4 planes [32 lanes][2]
//            (16 bytes a lane a plane: conflict-free 128-bit shared loads)
//   columns  NARROW: [32 lanes][8] bytes, then 8 int32 bases
//            WIDE: 2 planes [32 lanes][4] int32
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace fp {

constexpr int kCols = 8;          // SELL columns of a record

template <typename V, bool WIDE>
struct Record {
    static constexpr int val = kCols * 32 * (int)sizeof(V);
    static constexpr int idx = WIDE ? kCols * 32 * 4 : kCols * 32;
    static constexpr int bytes = val + idx + (WIDE ? 0 : kCols * 4);
    static_assert(bytes % 16 == 0, "bulk copies move multiples of 16 bytes");
};

// byte offset of entry (column j, lane) in a record's value section
template <typename V>
__host__ __device__ constexpr int record_value_at(int j, int lane) {
    return sizeof(V) == 4 ? ((j >> 2) * 32 + lane) * 16 + (j & 3) * 4 : ((j >> 1) * 32 + lane) * 16 + (j & 1) * 8;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_evict_normal() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar), "l"(policy)
        : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

constexpr int kMaxStages = 8;
constexpr int kStreamBars = 2 * kMaxStages;   // mbarriers of a warp: per stage one for its copy, one for its release
constexpr int kCopySpin = 1 << 20;   // polls of one mbarrier before the solve gives up (each poll suspends for a while)

// polls until the phase of that parity has completed; false when the bound ends the wait
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (int k = 0; k < kCopySpin; k++)
        if (mbar_try(bar, parity)) return true;
    return false;
}

// A warp's part of the matrix and its ring.  Copy number q of a stream (counted
// from begin) lands in stage q % stages and completes phase q / stages of that
// stage's first mbarrier; once the 32 lanes have read the stage they complete
// the same phase of its second mbarrier, and the next copy into it waits for
// that.  `stage` and `parity` track the next copy to consume, `inflight` the
// copies issued and not yet consumed.
struct WarpStream {
    uint32_t ring, bars;         // shared addresses of the warp's ring and its mbarriers
    int s0, s1;                  // slices [s0, s1)
    int rec0, nrec;              // records [rec0, rec0 + nrec) cover them
    int skip;                    // leading columns of the first record that belong to the slice before
    int stage, inflight;
    uint32_t parity;
    int next;                    // record (relative to rec0) the next copy fetches
    uint64_t policy;
};

// One record type streamed through a warp's ring of RING bytes.
template <typename V, bool WIDE, int RING>
struct Stream {
    using Rec = Record<V, WIDE>;
    static constexpr int stages = RING / Rec::bytes < kMaxStages ? RING / Rec::bytes : kMaxStages;
    static_assert(stages >= 2, "a ring holds at least two records");

    __device__ static uint32_t full(const WarpStream &w, int stage) { return w.bars + 8u * stage; }
    __device__ static uint32_t empty(const WarpStream &w, int stage) { return w.bars + 8u * (kMaxStages + stage); }

    // lane 0 fetches the next record into `stage`; `reused`: once the lanes have
    // released what the stage held (the phase of `parity`).  A release that does
    // not come within the bound leaves the copy out, and its consumer gives up.
    __device__ static void issue(WarpStream &w, const unsigned char *recs, int stage, bool reused, uint32_t parity) {
        if ((threadIdx.x & 31) == 0 && (!reused || mbar_wait(empty(w, stage), parity))) {
            mbar_expect(full(w, stage), Rec::bytes);
            bulk_load(w.ring + (uint32_t)stage * Rec::bytes, recs + (size_t)(w.rec0 + w.next) * Rec::bytes, Rec::bytes,
                      full(w, stage), w.policy);
        }
        __syncwarp();
        w.next = w.next + 1 == w.nrec ? 0 : w.next + 1;
        w.inflight++;
    }
    // sets the ring up and fills it from the first record on, with at most
    // `most` copies (nrec: a single pass follows)
    __device__ static void begin(WarpStream &w, const unsigned char *recs, int most) {
        w.next = w.stage = w.inflight = 0;
        w.parity = 0;
        if (w.nrec == 0) return;
        if ((threadIdx.x & 31) == 0) {
            for (int k = 0; k < stages; k++) {
                mbar_init(full(w, k), 1);
                mbar_init(empty(w, k), 32);
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        __syncwarp();
        for (int k = 0; k < stages && k < most; k++) issue(w, recs, k, false, 0);
    }
    // the copy of the next stage to consume has landed (the same answer in every lane)
    __device__ static bool wait(const WarpStream &w) {
        return __all_sync(0xFFFFFFFFu, mbar_wait(full(w, w.stage), w.parity));
    }
    __device__ static void step(WarpStream &w) {
        w.inflight--;
        if (++w.stage == stages) {
            w.stage = 0;
            w.parity ^= 1u;
        }
    }
    // waits for every copy in flight and releases the mbarriers (the ring may
    // then serve another stream, or the block may leave)
    __device__ static bool end(WarpStream &w) {
        if (w.nrec == 0) return true;
        bool ok = true;
        while (w.inflight > 0) {
            ok = wait(w) && ok;
            step(w);
        }
        __syncwarp();
        if ((threadIdx.x & 31) == 0)
            for (int k = 0; k < stages; k++) {
                asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(full(w, k)) : "memory");
                asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(empty(w, k)) : "memory");
            }
        __syncwarp();
        return ok;
    }
    // A record in registers: its values, and its entries' vector values on
    // their way
    struct Frag {
        V a[kCols], g[kCols];
    };
    // Loads the record of the next stage, releases the stage if a copy will
    // follow into it, and starts the record's gathers.  The release: every lane
    // orders its reads before the async proxy's writes and arrives on the
    // stage's second mbarrier, which lane 0 waits for before it issues the copy
    // (loads merely issued were seen overtaken by the copy).  It comes before
    // the gathers, so that lane 0 finds it complete.
    __device__ static void fetch(const WarpStream &w, const V *v, bool follows, Frag &f) {
        const int lane = threadIdx.x & 31;
        const uint32_t st = w.ring + (uint32_t)w.stage * Rec::bytes;
        int col[kCols];
        if constexpr (sizeof(V) == 4) {
#pragma unroll
            for (int h = 0; h < 2; h++)
                asm volatile("ld.volatile.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                             : "=f"(f.a[4 * h]), "=f"(f.a[4 * h + 1]), "=f"(f.a[4 * h + 2]), "=f"(f.a[4 * h + 3])
                             : "r"(st + 512u * h + 16u * lane));
        } else {
#pragma unroll
            for (int h = 0; h < 4; h++)
                asm volatile("ld.volatile.shared.v2.f64 {%0, %1}, [%2];"
                             : "=d"(f.a[2 * h]), "=d"(f.a[2 * h + 1])
                             : "r"(st + 512u * h + 16u * lane));
        }
        if constexpr (WIDE) {
#pragma unroll
            for (int h = 0; h < 2; h++)
                asm volatile("ld.volatile.shared.v4.s32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(col[4 * h]), "=r"(col[4 * h + 1]), "=r"(col[4 * h + 2]), "=r"(col[4 * h + 3])
                             : "r"(st + Rec::val + 512u * h + 16u * lane));
        } else {
            uint32_t lo, hi;
            asm volatile("ld.volatile.shared.v2.u32 {%0, %1}, [%2];" : "=r"(lo), "=r"(hi) : "r"(st + Rec::val + 8u * lane));
#pragma unroll
            for (int h = 0; h < 2; h++)
                asm volatile("ld.volatile.shared.v4.s32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(col[4 * h]), "=r"(col[4 * h + 1]), "=r"(col[4 * h + 2]), "=r"(col[4 * h + 3])
                             : "r"(st + Rec::val + Rec::idx + 16u * h));
#pragma unroll
            for (int j = 0; j < 4; j++) {
                col[j] += lane + (int)((lo >> (8 * j)) & 255u);
                col[4 + j] += lane + (int)((hi >> (8 * j)) & 255u);
            }
        }
        if (follows) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(empty(w, w.stage));
        }
#pragma unroll
        for (int j = 0; j < kCols; j++) f.g[j] = v[col[j]];
    }
    // One product over the warp's rows: fin(i, sum_j A_ij v_j, v_i), the sum in
    // column order.  width(sl): entries of a row of slice sl.  With `more` the
    // ring is kept full for the pass that follows; v, and every row the pass
    // hands to fin, are padded to whole slices (rows past the matrix have no
    // entries: their sums are 0).
    template <typename W, typename F>
    __device__ static bool pass(WarpStream &w, const unsigned char *recs, const V *v, bool more, W width, F fin) {
        if (w.nrec == 0) return true;
        const int lane = threadIdx.x & 31;
        int sl = w.s0, i = sl * 32 + lane;
        int rem = width(sl) + w.skip;
        V acc = 0, vi = v[i];
        auto next_row = [&](V total, V rest) {
            if (sl < w.s1) fin(i, total, vi);
            acc = rest;
            if (++sl < w.s1) {
                i += 32;
                rem = width(sl);
                vi = v[i];
            }
        };
        // three forms, the branches uniform: no slice ends in the record, one
        // does (after column rem - 1), or several short ones do
        auto sum = [&](const Frag &f) {
            if (rem > kCols) {
#pragma unroll
                for (int j = 0; j < kCols; j++) acc = fma(f.a[j], f.g[j], acc);
                rem -= kCols;
            } else if (rem > 0 && (sl + 1 >= w.s1 || rem + width(sl + 1) > kCols)) {
                const int e = rem - 1;
                V total = 0;
#pragma unroll
                for (int j = 0; j < kCols; j++) {
                    acc = fma(f.a[j], f.g[j], acc);
                    total = j == e ? acc : total;
                    acc = j == e ? (V)0 : acc;
                }
                next_row(total, acc);
                rem -= kCols - 1 - e;
            } else {
#pragma unroll
                for (int j = 0; j < kCols; j++) {
                    acc = fma(f.a[j], f.g[j], acc);
                    if (--rem == 0) next_row(acc, (V)0);
                }
            }
        };
        Frag f;
        for (int c = 0; c < w.nrec; c++) {
            if (!wait(w)) return false;
            const bool follows = more || c + stages < w.nrec;
            const int stage = w.stage;
            const uint32_t parity = w.parity;
            fetch(w, v, follows, f);
            step(w);
            if (follows) issue(w, recs, stage, true, parity);
            if (c == 0) {
#pragma unroll
                for (int j = 0; j < kCols; j++)
                    if (j < w.skip) f.a[j] = 0;
            }
            sum(f);
        }
        return true;
    }
};

}  // namespace fp
