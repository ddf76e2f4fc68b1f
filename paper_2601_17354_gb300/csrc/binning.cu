// K2 counts, K3 coarse entries, K4 radix sort, K5 tile lists and ranges.
//
// The pair lists carry the canonical index of each Gaussian: this is the permutation pi of Eq. 10
// ("a GPU sort yields a permutation mapping sorted index i to canonical index pi(i)").  Parameters
// are never reordered; the compositing kernels gather by pi and the backward scatters gradients to
// pi (index-mapped gradient scattering).
//
// Every tile's list holds the Gaussians that reach it in depth order, ties in canonical order: the
// order of the stable sort of (tile << 32 | depth bits) pairs.  It is built in two levels.  The
// Gaussians are sorted by depth (32-bit keys, ties kept in canonical order); each then emits one
// coarse entry per super-tile (kSuperW x kSuperH tiles) its tile rectangle overlaps, in depth
// order; a stable radix sort by super-tile id groups the entries by super-tile, still in depth
// order inside each group.  The fine stage gives each entry a 32-bit mask of the super-tile's tiles
// the Gaussian reaches (the projection's reach test), counts each tile's entries per block of
// kFineBlock (a warp's 32 masks transposed in five shuffle stages, so lane x holds the lanes that
// reach tile x), scans those counts, and writes each entry's canonical index at its tile's first
// pair + the entries of the tile before it.  The pair buffer is laid out
// super-tile by super-tile, tiles row-major inside; a tile's list is [ranges[t].x, ranges[t].y).
// The pair count is the sum of the projection's reached-tile counts, known before any list is
// built; pairs beyond the capacity are not written (the status word records the overflow and the
// capacity needed), so no host synchronisation sits between projection and compositing.
//
// The radix sort is least-significant-digit first, 8-bit digits, over the bits that can be
// non-zero (32 depth bits for the Gaussians, ceil(log2 super-tiles) bits for the coarse entries;
// the caller's low key bits of the 64-bit keys of the allocation-free entry point); the last digit
// is masked to what is left of the bit range.  The digit totals of every pass come from one
// up-front histogram; each pass is then one launch that ranks a tile's keys with warp ballots and
// finds the tile's place by decoupled look-back over the tiles before it (bounded waits, see
// k_onesweep).
//
// The kernels of a render's binning start with pdl_begin() and are launched by launch_pdl (the
// timeout self-test launches plainly): the next one is scheduled while the current one's last
// CTAs run and waits for them before it touches memory.
// The scratch these kernels expect zeroed (look-back words, digit totals, counters, ranges) is
// cleared by the projection before them (render_zero_plan), or by memsets when the caller says so.
#include "pgs_internal.cuh"

namespace pgs {
namespace {

constexpr unsigned kFull = 0xffffffffu;
static_assert(kSortThreads == kRadix, "one thread per digit in the sort kernels");

// ---------------------------------------------------------------------------------------------
// K2: pair count and coarse entry counts
// ---------------------------------------------------------------------------------------------
constexpr int kScanThreads = 1024;

// super-tile rectangle [sx0, sx1) x [sy0, sy1) of a tile rectangle (x0 | y0 << 16, x1 | y1 << 16)
__device__ __forceinline__ void super_rect(uint2 r, uint32_t& sx0, uint32_t& sy0, uint32_t& sx1, uint32_t& sy1) {
    sx0 = (r.x & 0xffffu) / kSuperW;
    sy0 = (r.x >> 16) / kSuperH;
    sx1 = ((r.y & 0xffffu) + kSuperW - 1) / kSuperW;
    sy1 = ((r.y >> 16) + kSuperH - 1) / kSuperH;
}

// Exclusive scan of `count` values by one CTA (a whole number of warps, at most 1024 threads),
// kV consecutive values per thread and step: load(i) gives value i, store(i, prefix) receives its
// exclusive prefix; returns the total to every thread.  Every thread of the CTA calls it.
template <class Load, class Store>
__device__ unsigned long long cta_scan(int count, Load load, Store store) {
    constexpr int kV = 8;
    __shared__ unsigned long long s_warp[32];
    __shared__ unsigned long long s_carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < count; base += blockDim.x * kV) {
        const int first = base + threadIdx.x * kV;
        unsigned long long v[kV], tsum = 0;
#pragma unroll
        for (int k = 0; k < kV; ++k) {
            v[k] = first + k < count ? load(first + k) : 0ull;
            tsum += v[k];
        }
        unsigned long long incl = tsum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const unsigned long long w = lane < nw ? s_warp[lane] : 0ull;
            unsigned long long wi = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long t = __shfl_up_sync(kFull, wi, o);
                if (lane >= o) wi += t;
            }
            if (lane < nw) s_warp[lane] = wi - w;
        }
        __syncthreads();
        const unsigned long long carry = s_carry;
        unsigned long long run = carry + s_warp[warp] + incl - tsum;
#pragma unroll
        for (int k = 0; k < kV; ++k) {
            if (first + k < count) store(first + k, run);
            run += v[k];
        }
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) s_carry = run;
        __syncthreads();
    }
    return s_carry;
}

// Is this CTA the last of the grid to get here?  Each CTA's writes before the call are visible to
// the last one (fence before the ticket, fence after); the last CTA resets the ticket.  No CTA
// waits for another.
__device__ __forceinline__ bool last_cta(uint32_t* ticket) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        if (s_last) *ticket = 0u;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

// Per block of kProjBlock depth-ordered Gaussians (the coarse emission's CTAs): coarse entries
// (super-tiles of the rectangle) into block_sums; reached tiles added into pair_count (zeroed
// before).  A CTA takes kCountItems such blocks, one Gaussian of each per thread, so each thread
// has that many independent gathers in flight.  The last CTA then scans the per-block counts into
// their offsets and sets the coarse total, the coarse sort's CTA count, the capacity the render
// needs (pairs, and the coarse stage's entries and counters) and the capacity check.
constexpr int kCountItems = 4;
__global__ void __launch_bounds__(kProjBlock)
k_coarse_counts(int64_t n, int64_t capacity, int64_t supers, const uint32_t* __restrict__ perm, Scratch sc) {
    pdl_begin();
    const int64_t nbk = (n + kProjBlock - 1) / kProjBlock;  // blocks of the emission
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t g[kCountItems], reached[kCountItems], area[kCountItems];
    uint2 rect[kCountItems];
#pragma unroll
    for (int k = 0; k < kCountItems; ++k) {
        const int64_t i = ((int64_t)blockIdx.x * kCountItems + k) * kProjBlock + threadIdx.x;
        g[k] = i < n ? perm[i] : 0xffffffffu;
    }
#pragma unroll
    for (int k = 0; k < kCountItems; ++k) {
        const bool valid = g[k] != 0xffffffffu;
        reached[k] = valid ? sc.touched[g[k]] : 0u;
        rect[k] = valid ? sc.rect[g[k]] : make_uint2(0u, 0u);
    }
    __shared__ uint32_t s_a[kCountItems][kProjBlock / 32], s_r[kProjBlock / 32];
    uint32_t rsum = 0;
#pragma unroll
    for (int k = 0; k < kCountItems; ++k) {
        area[k] = 0;
        if (reached[k]) {
            uint32_t sx0, sy0, sx1, sy1;
            super_rect(rect[k], sx0, sy0, sx1, sy1);
            area[k] = (sx1 - sx0) * (sy1 - sy0);
        }
        const uint32_t wa = __reduce_add_sync(kFull, area[k]);
        if (lane == 0) s_a[k][warp] = wa;
        rsum += reached[k];
    }
    const uint32_t wr = __reduce_add_sync(kFull, rsum);
    if (lane == 0) s_r[warp] = wr;
    __syncthreads();
    if (threadIdx.x < 32) {
        const bool in = threadIdx.x < kProjBlock / 32;
#pragma unroll
        for (int k = 0; k < kCountItems; ++k) {
            const uint32_t a = __reduce_add_sync(kFull, in ? s_a[k][threadIdx.x] : 0u);
            const int64_t b = (int64_t)blockIdx.x * kCountItems + k;
            if (threadIdx.x == 0 && b < nbk) sc.block_sums[b] = a;
        }
        const unsigned long long r = __reduce_add_sync(kFull, in ? s_r[threadIdx.x] : 0u);
        if (threadIdx.x == 0 && r) atomicAdd(sc.pair_count, r);
    }
    if (!last_cta(&sc.bin_ticket[0])) return;
    const unsigned long long Ce = cta_scan(
        (int)nbk, [&](int k) { return (unsigned long long)__ldcg(&sc.block_sums[k]); },
        [&](int k, unsigned long long v) { sc.block_offsets[k] = v; });
    if (threadIdx.x == 0) {
        const unsigned long long P = atomicAdd(sc.pair_count, 0ull);
        *sc.coarse_count = Ce;
        const unsigned long long kept = Ce < (unsigned long long)capacity ? Ce : (unsigned long long)capacity;
        *sc.sort_blocks = (uint32_t)((kept + kSortTile - 1) / kSortTile);
        const unsigned long long c = coarse_need(Ce, (unsigned long long)supers);
        const unsigned long long need = P > c ? P : c;
        *sc.pair_need = need;
        if (need > (unsigned long long)capacity) atomicOr(sc.status, kStatusCapacity);
    }
}

// Transpose of the warp's 32 x 32 bit matrix (lane l holds row l): lane x returns column x, whose
// bit l is bit x of lane l's word.  Five stages; at stage j the lanes l and l ^ j swap the block of
// bits b with b & j set (upper lane l) against the block with b & j clear (lower lane l ^ j).
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x, int lane) {
    constexpr uint32_t kMask[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const int j = 16 >> k;
        const uint32_t m = kMask[k];
        const uint32_t o = __shfl_xor_sync(kFull, x, j);
        x = (lane & j) ? ((x & ~m) | ((o & ~m) >> j)) : ((x & m) | ((o & m) << j));
    }
    return x;
}

// Reach masks of entries without one of the projection's (rectangles of more than 32 tiles over more than 2 x 2
// super-tiles), warp-collective: tiles of the super-tile at tile (bx, by) (each lane its own) that Gaussian g
// reaches, bit (ty - by) kSuperW + tx - bx; 0 for lanes without `need`.  The warp runs the projection's
// reach test over all such lanes' candidate tiles together, 32 per round (candidate k by lane k mod 32), so one
// large Gaussian does not hold its warp for 32 tests.
struct BigSmem {
    uint32_t mask[32], lane[32];
    uint4 cand[32];  // first candidate, tile x0 | y0 << 16 of the part inside the super-tile, its width, Gaussian
};
__device__ __forceinline__ uint32_t entry_mask(bool need, uint32_t g, uint2 r, uint32_t bx, uint32_t by, int T,
                                               const Scratch& sc, int lane, BigSmem& S) {
    if (!__any_sync(kFull, need)) return 0u;
    uint32_t X0 = 0, Y0 = 0, w = 0, ncand = 0;
    if (need) {
        X0 = max(r.x & 0xffffu, bx);
        Y0 = max(r.x >> 16, by);
        w = min(r.y & 0xffffu, bx + kSuperW) - X0;  // >= 1: the super-tile lies in the Gaussian's super-tile rectangle
        ncand = w * (min(r.y >> 16, by + kSuperH) - Y0);
    }
    WarpRuns runs(ncand);
    S.mask[lane] = 0u;
    if (need) {
        S.lane[runs.rank] = (uint32_t)lane;
        S.cand[runs.rank] = make_uint4(runs.first, X0 | (Y0 << 16), w, g);
    }
    __syncwarp();
    for (uint32_t b = 0; b < runs.total; b += 32) {
        const uint32_t o = runs.owner(b), k = b + (uint32_t)lane;
        if (k < runs.total) {
            const uint4 c = S.cand[o];
            const uint32_t local = k - c.x, dy = local / c.z, dx = local - dy * c.z;
            const uint32_t tx = (c.y & 0xffffu) + dx, ty = (c.y >> 16) + dy;
            const float4 p = sc.xyo[c.w], q = sc.conic[c.w];
            if (tile_hit(p.x, p.y, q.x, q.y, q.z, __fdiv_rn(q.y, q.x), __fdiv_rn(q.y, q.z), (int)tx, (int)ty, (float)T))
                atomicOr(&S.mask[S.lane[o]], 1u << ((ty % kSuperH) * kSuperW + tx % kSuperW));
        }
    }
    __syncwarp();
    return S.mask[lane];
}

// ---------------------------------------------------------------------------------------------
// K3: coarse entries of one CTA's Gaussians in depth order, super-tiles row-major inside each
// Gaussian's super-tile rectangle: key = super-tile id, value = the entry's own position e0, and at
// e0 the Gaussian's canonical index and its reach mask of the super-tile (rectangles of <= 32
// tiles: read from their reach bits; larger ones whose super-tile rectangle spans at most 2 x 2:
// the projection's masks; the rest: entry_mask).  Each warp walks
// the entries of its own 32 Gaussians, 32 per round (entry k by lane k mod 32), whose records it
// keeps in shared memory by rank.  kEmitWarps warps share the rounds of 32 Gaussians: a round is one
// chain of dependent steps, and 100k Gaussians are only five warps to each scheduler.  Four where the grid
// leaves the SMs fewer than four CTAs each, one elsewhere: 100k Gaussians at 1280x720 with 8-pixel tiles (391
// CTAs) 38 us with one, 26 with two, 22 with four; 200k with 16-pixel tiles (782 CTAs) lose 1 and 10 us
// a step with two and four, 500k 5 and 25 us (the set-up is most of their work).
// ---------------------------------------------------------------------------------------------
struct CoarseRec {
    uint4 a;  // rectangle, hitmask, Gaussian
    uint4 b;  // first entry, super-tiles across | how << 30, super-tiles of a row of the grid, first super-tile
    uint4 m;  // the projection's masks (how = 0), else 1 / super-tiles across (a float)
};
template <int kEmitWarps>
__global__ void __launch_bounds__(kProjBlock * kEmitWarps)
k_coarse_emit(int64_t n, int SX, int T, int64_t capacity, const uint32_t* __restrict__ perm, Scratch sc,
              uint32_t* __restrict__ gidx, uint32_t* __restrict__ gmask, int passes, uint32_t last_mask,
              const RenderDesc* __restrict__ renders, int R) {
    pdl_begin();
    __shared__ CoarseRec s_rec[kProjBlock];
    __shared__ uint32_t s_cnt[kProjBlock], s_warp[kProjBlock / 32];
    __shared__ BigSmem s_big[kProjBlock * kEmitWarps / 32];
    __shared__ uint32_t s_hist[4][kRadix];  // digit counts of the written keys, pass by pass
    const int t = threadIdx.x, lane = t & 31, warp = (t & (kProjBlock - 1)) >> 5, part = t / kProjBlock;
    const int64_t i = (int64_t)blockIdx.x * kProjBlock + t;
    for (int k = t; k < passes * kRadix; k += kProjBlock * kEmitWarps) (&s_hist[0][0])[k] = 0u;
    CoarseRec* const recs = s_rec + 32 * warp;
    if (part == 0) {
        // the Gaussian's record in one memory latency (what a culled one holds there is not used)
        const uint32_t g = i < n ? perm[i] : 0u;
        const uint2 r = i < n ? sc.rect[g] : make_uint2(0u, 0u);
        const uint32_t hm = i < n ? sc.hitmask[g] : 0u;
        const uint32_t reached = i < n ? sc.touched[g] : 0u;
        uint32_t cnt = 0, w = 1, how = 0;
        if (reached) {
            uint32_t sx0, sy0, sx1, sy1;
            super_rect(r, sx0, sy0, sx1, sy1);
            w = sx1 - sx0;
            cnt = w * (sy1 - sy0);
            const uint32_t area = ((r.y & 0xffffu) - (r.x & 0xffffu)) * ((r.y >> 16) - (r.x >> 16));
            how = area <= 32u ? 1u : w <= 2u && sy1 - sy0 <= 2u ? 0u : 2u;  // hitmask, the projection's masks, entry_mask
        }
        s_cnt[t] = cnt;
        const WarpRuns runs(cnt);
        if (reached) {
            CoarseRec& o = recs[runs.rank];
            o.a = make_uint4(r.x, r.y, hm, g);
            uint32_t sx = (uint32_t)SX, first_super = 0;
            if (renders) {  // batch: item g belongs to the last render whose first item is <= g
                int lo = 0, hi = R - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (renders[mid].item_base <= (int64_t)g) lo = mid;
                    else hi = mid - 1;
                }
                sx = (uint32_t)renders[lo].SX;
                first_super = (uint32_t)renders[lo].super_base;
            }
            o.b = make_uint4(runs.first, w | (how << 30), sx, first_super);
            if (how == 0u) o.m = sc.smask[g];
            else o.m.x = __float_as_uint(__frcp_rn((float)w));
        }
        if (lane == 0) s_warp[warp] = runs.total;
    }
    __syncthreads();
    const WarpRuns runs(s_cnt[32 * warp + lane]);
    uint32_t before = 0;
#pragma unroll
    for (int k = 0; k < kProjBlock / 32; ++k) before += k < warp ? s_warp[k] : 0u;
    const unsigned long long out = sc.block_offsets[blockIdx.x] + before;
    uint32_t* ck = reinterpret_cast<uint32_t*>(sc.keys[0]);
    for (uint32_t b = 32 * part; b < runs.total; b += 32 * kEmitWarps) {  // warp-uniform
        const uint32_t k = b + (uint32_t)lane;
        const CoarseRec& o = recs[runs.owner(b)];
        const bool valid = k < runs.total;
        const uint4 ra = o.a, rb = o.b;
        const uint32_t ow = rb.y & 0x3fffffffu, kind = valid ? rb.y >> 30 : 3u;
        const uint4 rm = o.m;
        const uint32_t local = k - rb.x;
        const uint32_t dy = kind == 0u ? local >> (ow - 1u)
                                       : local < 1024u ? small_quotient(local, __uint_as_float(rm.x)) : local / ow;
        const uint32_t dx = local - dy * ow;
        const uint32_t sx = (ra.x & 0xffffu) / kSuperW + dx, sy = (ra.x >> 16) / kSuperH + dy;
        const uint2 rect = make_uint2(ra.x, ra.y);
        uint32_t mask = entry_mask(kind == 2u, ra.w, rect, sx * kSuperW, sy * kSuperH, T, sc, lane, s_big[t >> 5]);
        if (kind == 1u)
            mask = super_mask_from_hits(ra.z, rect.x & 0xffffu, rect.x >> 16, rect.y & 0xffffu, rect.y >> 16, sx, sy);
        else if (kind == 0u)
            mask = smask_slot(rm, 2u * dy + dx);
        const unsigned long long pos = out + k;
        if (valid && pos < (unsigned long long)capacity) {
            const uint32_t key = rb.w + sy * rb.z + sx;
            ck[pos] = key;
            sc.vals[0][pos] = (uint32_t)pos;
            gidx[pos] = ra.w;
            gmask[pos] = mask;
            for (int p = 0; p < passes; ++p)
                atomicAdd(&s_hist[p][(key >> (p * kRadixBits)) & (p == passes - 1 ? last_mask : kRadix - 1)], 1u);
        }
    }
    // the sort's digit totals: this CTA's counts added into its partial copy (zeroed before)
    __syncthreads();
    uint32_t* copy = sc.digit_totals + (blockIdx.x % kTotalCopies) * (kMaxPasses * kRadix);
    for (int k = t; k < passes * kRadix; k += kProjBlock * kEmitWarps) {
        const uint32_t v = (&s_hist[0][0])[k];
        if (v) atomicAdd(&copy[k], v);
    }
}

// ---------------------------------------------------------------------------------------------
// K4: radix sort
// ---------------------------------------------------------------------------------------------

__device__ __forceinline__ uint64_t kept_pairs(const Scratch& sc, int64_t capacity) {
    const unsigned long long P = *sc.pair_count;
    return P < (unsigned long long)capacity ? P : (unsigned long long)capacity;
}

// digit totals of every pass (digits from bit first_shift up) in one read of the keys, added into
// the partial copy of the CTA
template <typename KeyT>
__global__ void __launch_bounds__(kSortThreads)
k_digit_totals(int64_t capacity, int first_shift, int passes, uint32_t last_mask, const KeyT* __restrict__ keys,
               Scratch sc) {
    pdl_begin();
    __shared__ uint32_t h[kMaxPasses][kRadix];
    for (int k = threadIdx.x; k < kMaxPasses * kRadix; k += kSortThreads) (&h[0][0])[k] = 0;
    __syncthreads();
    const uint64_t P = kept_pairs(sc, capacity);
    for (uint64_t k = (uint64_t)blockIdx.x * kSortThreads + threadIdx.x; k < P;
         k += (uint64_t)gridDim.x * kSortThreads) {
        const unsigned long long key = keys[k];
        for (int p = 0; p < passes; ++p)
            atomicAdd(&h[p][(key >> (first_shift + p * kRadixBits)) & (p == passes - 1 ? last_mask : kRadix - 1)], 1u);
    }
    __syncthreads();
    uint32_t* copy = sc.digit_totals + (blockIdx.x % kTotalCopies) * (kMaxPasses * kRadix);
    for (int k = threadIdx.x; k < passes * kRadix; k += kSortThreads) {
        const uint32_t v = (&h[0][0])[k];
        if (v) atomicAdd(&copy[k], v);
    }
}

// One pass of the sort in one launch (decoupled look-back): a CTA takes the next tile of
// kSortThreads x kItems keys from a ticket (so every tile before it belongs to a CTA already
// running), counts its keys per digit in shared memory and publishes those counts at once, so the
// tiles after it can add them up before it has finished.  It then ranks its keys by the pass's
// digit (per 32 consecutive keys the lanes of equal digit from one ballot per digit bit, warp
// prefixes per digit) and adds up the counts of the tiles before it by walking back until a tile
// that has published its inclusive prefix.  Each wait on a tile that has not published yet is
// bounded: past kSpinLimit polls (about a second) the CTA records kStatusTimeout, raises the sort's
// abort word, which ends every other wait at once, and leaves its keys unwritten.  The keys are
// then reordered by digit in shared memory and each digit's run written to its global offset
// (digits of smaller value from the pass's totals + the run of the tiles before), so the global
// writes are contiguous runs.
//
// Look-back words: value | flag << 30, flag 1 = the tile's own count, 2 = inclusive prefix of the
// tiles up to it; 0 = not yet published (the region is cleared before every sort).
constexpr uint32_t kLbCount = 1u << 30, kLbPrefix = 2u << 30, kLbValue = (1u << 30) - 1u;
constexpr int kSpinLimit = 1 << 20;  // with the back-off below, about half a second
constexpr int kLbWindow = 8;
constexpr int kDigitWarps = kRadix / 32;  // the warps whose threads own one digit each

// named barrier of the digit warps (the first kRadix threads); barrier 0 is __syncthreads
__device__ __forceinline__ void digit_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kRadix) : "memory"); }

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

template <typename KeyT, int kItems, int kThreads = kSortThreads>
constexpr size_t scatter_smem() { return (sizeof(KeyT) + sizeof(uint32_t)) * kThreads * kItems; }

// kThreads = kRadix or a multiple of it: with more threads than digits each warp ranks fewer keys
// and only the first kRadix threads take the per-digit steps (their own named barrier)
template <typename KeyT, int kItems, int kThreads = kSortThreads>
__global__ void __launch_bounds__(kThreads)
k_onesweep(int64_t capacity, int pass, int shift, uint32_t dmask, int sb_max, bool spare, const KeyT* __restrict__ kin,
           const uint32_t* __restrict__ vin, KeyT* __restrict__ kout, uint32_t* __restrict__ vout, Scratch sc) {
    pdl_begin();
    static_assert(kThreads % kRadix == 0, "whole digit warps");
    constexpr int kWarps = kThreads / 32;
    constexpr int kTile = kThreads * kItems;            // keys per CTA
    constexpr int kWarpItems = kTile / kWarps;          // contiguous keys per warp
    constexpr int kRounds = kWarpItems / 32;            // == kItems
    extern __shared__ __align__(16) unsigned char s_dyn[];
    KeyT* s_keys = reinterpret_cast<KeyT*>(s_dyn);
    uint32_t* s_vals = reinterpret_cast<uint32_t*>(s_dyn + sizeof(KeyT) * kTile);
    __shared__ uint32_t s_wh[kWarps][kRadix];      // per-warp digit counts, then warp prefixes
    __shared__ uint32_t s_gofs[kRadix];            // global offset of this tile's run of digit d
    __shared__ uint32_t s_bstart[kRadix];          // start of digit d inside the CTA's reordering
    __shared__ uint32_t s_part[kDigitWarps];
    __shared__ uint32_t s_hist[kRadix];            // the tile's count of digit d
    __shared__ uint32_t s_tile;
    __shared__ int s_gone;  // a wait ran out
    uint32_t* head = sc.sort_hist;  // [0] abort word, [1 + pass] ticket of the pass, then the look-back
    uint32_t* lb = sc.sort_hist + kLookbackHead + (size_t)pass * kRadix * sb_max;
    // A pass over few tiles is a chain of memory latencies, so everything it reads is asked for at once: the
    // digit totals (needed last), and the keys of the tile that the ticket most likely names (CTAs are started in
    // order).  2,000 keys took 9.6 us a pass with each waiting for the one before, 7.4 us now; 500k
    // keys 13.5 us, 12.6 us.  A grid sized for the capacity has CTAs to spare (eight in nine of the 2,395 for the
    // super-tile sort of 500k Gaussians): those leave first, the tiles are for the others.
    const uint32_t nblk = *sc.sort_blocks;
    if (spare && blockIdx.x >= nblk) return;
    if (threadIdx.x == 0) s_tile = atomicAdd(&head[1 + pass], 1u);
    const uint64_t P = kept_pairs(sc, capacity);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    KeyT key[kRounds];
    uint32_t val[kRounds];
    uint32_t dr[kRounds];  // digit | warp-local rank << 8
    auto load_tile = [&](uint32_t t) {
#pragma unroll
        for (int r = 0; r < kRounds; ++r) {
            const uint64_t idx = (uint64_t)t * kTile + (uint64_t)warp * kWarpItems + (uint64_t)r * 32 + lane;
            const bool valid = idx < P;
            key[r] = valid ? kin[idx] : (KeyT)0;
            val[r] = valid ? vin[idx] : 0u;
        }
    };
    load_tile(blockIdx.x);
    uint32_t total[kTotalCopies];
    if (threadIdx.x < kRadix) {
#pragma unroll
        for (int cpy = 0; cpy < kTotalCopies; ++cpy)
            total[cpy] = sc.digit_totals[pass * kRadix + (size_t)cpy * kMaxPasses * kRadix + threadIdx.x];
    }
    for (int k = threadIdx.x; k < kWarps * kRadix; k += kThreads) (&s_wh[0][0])[k] = 0;
    if (threadIdx.x < kRadix) s_hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_gone = 0;
    __syncthreads();
    const uint32_t tile = s_tile;
    if (tile >= nblk) return;
    if (tile != blockIdx.x) load_tile(tile);
    const uint64_t cbase = (uint64_t)tile * kTile;
    const uint64_t wbase = cbase + (uint64_t)warp * kWarpItems;
    // the tile's digit counts, published before the ranking
#pragma unroll
    for (int r = 0; r < kRounds; ++r)
        if (wbase + (uint64_t)r * 32 + lane < P) atomicAdd(&s_hist[(uint32_t)(key[r] >> shift) & dmask], 1u);
    __syncthreads();
    uint32_t* const mine = lb + (size_t)tile * kRadix + (threadIdx.x & (kRadix - 1));
    if (threadIdx.x < kRadix) st_relaxed(mine, (tile == 0 ? kLbPrefix : kLbCount) | s_hist[threadIdx.x]);
    const int nbits = __popc(dmask);  // dmask = 2^bits - 1: higher digit bits are zero
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        const uint64_t idx = wbase + (uint64_t)r * 32 + lane;
        const bool valid = idx < P;
        const uint32_t d = valid ? (uint32_t)(key[r] >> shift) & dmask : 0u;
        // lanes holding the same digit: one ballot per digit bit (and one for validity)
        unsigned peers = __ballot_sync(kFull, valid);
        if (!valid) peers = ~peers;
#pragma unroll
        for (int b = 0; b < kRadixBits; ++b) {
            if (b >= nbits) break;  // warp-uniform
            const bool bit = (d >> b) & 1u;
            const unsigned bal = __ballot_sync(kFull, bit);
            peers &= bit ? bal : ~bal;
        }
        uint32_t before = 0;
        if (valid) before = s_wh[warp][d];
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) s_wh[warp][d] = before + __popc(peers);
        __syncwarp();
        dr[r] = valid ? (d | ((before + __popc(peers & lt)) << 8)) : 0xffffffffu;
    }
    __syncthreads();
    if (threadIdx.x < kRadix) {  // thread = digit: warp prefixes, the tile's count of the digit, its look-back
        const int d = threadIdx.x;
        uint32_t acc = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t cnt = s_wh[w][d];
            s_wh[w][d] = acc;
            acc += cnt;
        }
        uint32_t before = 0;  // keys of digit d in the tiles before this one
        if (tile != 0) {
            // kLbWindow predecessors per round, loaded together: the walk over tiles that have
            // published only their count costs one memory latency per window, not per tile
            int spins = 0;
            bool gone = false;
            int64_t t = (int64_t)tile - 1;
            while (t >= 0) {
                uint32_t w[kLbWindow];
#pragma unroll
                for (int k = 0; k < kLbWindow; ++k) w[k] = t - k >= 0 ? ld_relaxed(lb + (size_t)(t - k) * kRadix + d) : kLbPrefix;
                int k = 0;
                bool found = false;
#pragma unroll
                for (; k < kLbWindow; ++k) {
                    const uint32_t flag = w[k] & ~kLbValue;
                    if (flag == 0u) break;  // tile t - k has not published yet
                    before += w[k] & kLbValue;
                    if (flag == kLbPrefix) {
                        found = true;
                        break;
                    }
                }
                if (found) break;
                t -= k;
                if (k == kLbWindow) continue;
                // wait (bounded) for tile t, then take the next window from it
                while ((ld_relaxed(lb + (size_t)t * kRadix + d) & ~kLbValue) == 0u) {
                    if (++spins > kSpinLimit) {
                        atomicOr(sc.status, kStatusTimeout);
                        st_relaxed(head, 1u);
                        break;
                    }
                    if ((spins & 63) == 0 && ld_relaxed(head) != 0u) break;  // another wait ran out
                    __nanosleep(64);
                }
                if (ld_relaxed(head) != 0u) {
                    gone = true;
                    break;
                }
            }
            if (gone) s_gone = 1;  // and no prefix: the tiles after this one end at the same wait
            else st_relaxed(mine, kLbPrefix | (before + acc));
        }
        // offset of digit d in the pass's output: all keys of smaller digits + the tiles before
        uint32_t all = 0;
#pragma unroll
        for (int cpy = 0; cpy < kTotalCopies; ++cpy) all += total[cpy];
        uint32_t incl_all = all, incl = acc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t ta = __shfl_up_sync(kFull, incl_all, o), tb = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) {
                incl_all += ta;
                incl += tb;
            }
        }
        if (lane == 31) s_part[warp] = incl_all;
        digit_sync();
        uint32_t wpre = 0;
#pragma unroll
        for (int w = 0; w < kDigitWarps; ++w) wpre += w < warp ? s_part[w] : 0u;
        s_gofs[d] = wpre + incl_all - all + before;
        digit_sync();
        if (lane == 31) s_part[warp] = incl;  // the tile's own digit counts, for its reordering
        digit_sync();
        wpre = 0;
#pragma unroll
        for (int w = 0; w < kDigitWarps; ++w) wpre += w < warp ? s_part[w] : 0u;
        s_bstart[d] = wpre + incl - acc;
    }
    __syncthreads();
    if (s_gone) return;  // a wait of this tile ran out: its keys stay where they were (status recorded)
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        if (dr[r] != 0xffffffffu) {
            const uint32_t d = dr[r] & 0xffu;
            const uint32_t pos = s_bstart[d] + s_wh[warp][d] + (dr[r] >> 8);
            if (pos < (uint32_t)kTile) {
                s_keys[pos] = key[r];
                s_vals[pos] = val[r];
            } else {
                atomicOr(sc.status, kStatusInternal);
            }
        }
    }
    __syncthreads();
    const uint32_t count = (uint32_t)min((uint64_t)kTile, P - cbase);
    for (uint32_t p = threadIdx.x; p < count; p += kThreads) {
        const KeyT k = s_keys[p];
        const uint32_t d = (uint32_t)(k >> shift) & dmask;
        const uint64_t dst = (uint64_t)s_gofs[d] + (p - s_bstart[d]);
        if (dst < P) {
            kout[dst] = k;
            vout[dst] = s_vals[p];
        } else {
            atomicOr(sc.status, kStatusInternal);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// K5: tile ranges [first, last + 1) from the sorted keys (ranges pre-zeroed)
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k_ranges(int64_t capacity, uint32_t tiles, const uint32_t* __restrict__ keys, Scratch sc) {
    pdl_begin();
    const uint64_t P = kept_pairs(sc, capacity);
    // four consecutive keys per thread step (one 16-byte load), with the neighbours either side
    for (uint64_t k0 = ((uint64_t)blockIdx.x * 256 + threadIdx.x) * 4; k0 < P; k0 += (uint64_t)gridDim.x * 1024) {
        uint32_t t[6];
        t[0] = k0 > 0 ? keys[k0 - 1] : 0xffffffffu;
        if (k0 + 4 <= P) {
            const uint4 q = *reinterpret_cast<const uint4*>(keys + k0);
            t[1] = q.x;
            t[2] = q.y;
            t[3] = q.z;
            t[4] = q.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) t[1 + j] = k0 + j < P ? keys[k0 + j] : 0xffffffffu;
        }
        t[5] = k0 + 4 < P ? keys[k0 + 4] : 0xffffffffu;
#pragma unroll
        for (int j = 1; j <= 4; ++j) {
            const uint64_t k = k0 + j - 1;
            if (k >= P) break;
            if (t[j] >= tiles) {
                atomicOr(sc.status, kStatusInternal);
                continue;
            }
            if (t[j - 1] != t[j]) sc.ranges[t[j]].x = (uint32_t)k;
            if (t[j + 1] != t[j]) sc.ranges[t[j]].y = (uint32_t)(k + 1);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// K5: fine stage.  The coarse entries of a super-tile, in depth order, are cut into blocks of
// kFineBlock; a block computes each entry's 32-bit mask of reached tiles of the super-tile and its
// per-tile counts; a scan over each super-tile's blocks and one over the super-tiles give every
// (block, tile) its first pair, and the block writes its pairs: entry e of tile x goes after the
// entries of x in earlier blocks, earlier warps and earlier lanes, i.e. in depth order.
// ---------------------------------------------------------------------------------------------
constexpr int kFineThreads = 256;
constexpr int kFineWarps = kFineThreads / 32;
constexpr int kFineRounds = kFineBlock / kFineThreads;  // entries per thread: warp w takes the
                                                        // block's entries [64 w, 64 w + 64), 32 a round
constexpr int kFineGrid = 152 * 8;  // grid-stride over the blocks

// tile grid of super-tile s: its position and the render it belongs to
struct SuperCell {
    uint32_t sx, sy;
    int TX, TY;
    uint32_t tile_base;
};

__device__ __forceinline__ SuperCell super_cell(uint32_t s, int TX, int TY, const RenderDesc* __restrict__ renders,
                                                int R) {
    SuperCell c;
    uint32_t local = s, SX = (uint32_t)((TX + kSuperW - 1) / kSuperW);
    c.TX = TX;
    c.TY = TY;
    c.tile_base = 0;
    if (renders) {  // the last render whose first super-tile is <= s
        int lo = 0, hi = R - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (renders[mid].super_base <= (int64_t)s) lo = mid;
            else hi = mid - 1;
        }
        local = s - (uint32_t)renders[lo].super_base;
        SX = (uint32_t)renders[lo].SX;
        c.TX = renders[lo].TX;
        c.TY = renders[lo].TY;
        c.tile_base = (uint32_t)renders[lo].tile_base;
    }
    c.sy = local / SX;
    c.sx = local - c.sy * SX;
    return c;
}

// tile of the image at bit x of super-tile c's masks, or -1
__device__ __forceinline__ int64_t tile_of_bit(const SuperCell& c, uint32_t x) {
    const uint32_t tx = c.sx * kSuperW + x % kSuperW, ty = c.sy * kSuperH + x / kSuperW;
    return (int)tx < c.TX && (int)ty < c.TY ? (int64_t)c.tile_base + ty * (uint32_t)c.TX + tx : -1;
}

// The compositing schedule, heaviest tiles first: a counting sort of the tiles into 128 quarter-octave
// buckets of their list length (only the schedule depends on it, never a result; the order inside a
// bucket is arbitrary).  k_seg_scan, which has the lengths, counts the buckets and its last CTA scans the counts;
// k_fine_emit puts the tiles down.  (As a kernel of its own the sort was one CTA, or three launches for
// more than 16,384 tiles: 12 us at 1920x1080, 17 us for the 14,400 8-pixel tiles of 1280x720.)
constexpr int kOrderBuckets = 128;
__device__ __forceinline__ int order_bucket(uint32_t len) {
    // lengths 0..3 are their own buckets; from 4 on, 4 (l - 1) + the two bits after the leading
    // one (l = floor(log2 len)): monotone in the length, at most 123
    int b = (int)len;
    if (len >= 4) {
        const int l = 31 - __clz(len);
        b = 4 * (l - 1) + (int)((len >> (l - 2)) & 3u);
    }
    return kOrderBuckets - 1 - b;
}

// One added to a bucket's counter for each lane of the warp with a tile (the lanes of a bucket, neighbouring tiles
// of similar length, by one atomic); returns the lane's place.
__device__ __forceinline__ uint32_t bucket_add(uint32_t* counters, bool has, uint32_t len) {
    const int lane = threadIdx.x & 31, b = has ? order_bucket(len) : -1;
    const unsigned same = __match_any_sync(kFull, b);
    const int leader = __ffs(same) - 1;
    uint32_t first = 0;
    if (has && lane == leader) first = atomicAdd(&counters[b], (uint32_t)__popc(same));
    return __shfl_sync(kFull, first, leader) + __popc(same & ((1u << lane) - 1u));
}

// One CTA: blocks per super-tile (ceil(entries / kFineBlock)), their exclusive scan into vbase
// (vbase[S] = all blocks) and each block's record binfo[v] = (super-tile, first entry, end entry,
// block index inside the super-tile).
// crange_from: 0 = crange is already filled (k_ranges over the sorted keys); 1 = the sort was one
// pass of the whole super-tile id (S <= 256): crange is the exclusive scan of its digit totals;
// 2 = one super-tile: crange[0] = all kept entries.
__global__ void __launch_bounds__(kScanThreads)
k_block_prefix(int S, int64_t capacity, Scratch sc, int crange_from) {
    pdl_begin();
    __shared__ uint32_t s_warp[kScanThreads / 32];
    __shared__ uint32_t s_carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (crange_from == 1) {  // S <= 256 (the parameter is the same for every thread)
        const int s = threadIdx.x;
        uint32_t c = 0;
        if (s < kRadix) {
#pragma unroll
            for (int cpy = 0; cpy < kTotalCopies; ++cpy) c += sc.digit_totals[(size_t)cpy * kMaxPasses * kRadix + s];
        }
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        uint32_t before = 0;
        for (int w = 0; w < warp; ++w) before += s_warp[w];
        if (s < S) sc.crange[s] = make_uint2(before + incl - c, before + incl);
        __syncthreads();  // s_warp is reused below; crange is read below
    }
    if (crange_from == 2 && threadIdx.x == 0) {
        const unsigned long long Ce = *sc.coarse_count;
        sc.crange[0] = make_uint2(0u, (uint32_t)(Ce < (unsigned long long)capacity ? Ce : (unsigned long long)capacity));
    }
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < S; base += kScanThreads) {
        const int s = base + threadIdx.x;
        uint32_t nb = 0;
        if (s < S) {
            const uint2 cr = sc.crange[s];
            nb = (cr.y - cr.x + kFineBlock - 1) / kFineBlock;
        }
        uint32_t incl = nb;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const uint32_t w = s_warp[lane];
            uint32_t wi = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, wi, o);
                if (lane >= o) wi += t;
            }
            s_warp[lane] = wi - w;
        }
        __syncthreads();
        const uint32_t carry = s_carry;
        const uint32_t first = carry + s_warp[warp] + incl - nb;
        if (s < S) {
            sc.vbase[s] = first;
            const uint2 cr = sc.crange[s];
            for (uint32_t k = 0; k < nb; ++k)
                if (first + k < (uint64_t)capacity / 32)
                    sc.binfo[first + k] = make_uint4((uint32_t)s, cr.x + k * kFineBlock,
                                                     min(cr.x + (k + 1) * kFineBlock, cr.y), k);
        }
        __syncthreads();
        if (threadIdx.x == kScanThreads - 1) s_carry = carry + s_warp[warp] + incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) sc.vbase[S] = s_carry;
}

// Each block's per-tile counts wc[32 v + x] from its entries' masks.
__global__ void __launch_bounds__(kFineThreads)
k_fine_count(int64_t capacity, const uint32_t* __restrict__ cv, const uint32_t* __restrict__ gmask,
             uint32_t* __restrict__ wc, int S, Scratch sc) {
    pdl_begin();
    __shared__ uint32_t s_cw[kFineWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t VB = sc.vbase[S];
    for (uint32_t v = blockIdx.x; v < VB; v += gridDim.x) {
        if ((uint64_t)v >= (uint64_t)capacity / 32) break;  // no slot for the block (capacity status raised)
        const uint4 bi = sc.binfo[v];  // super-tile, first entry, end entry, block of the super-tile
        uint32_t m[kFineRounds];
#pragma unroll
        for (int r = 0; r < kFineRounds; ++r) {
            const uint64_t e = (uint64_t)bi.y + warp * (32 * kFineRounds) + r * 32 + lane;
            m[r] = e < bi.z ? gmask[cv[e]] : 0u;
        }
        uint32_t cnt = 0;
#pragma unroll
        for (int r = 0; r < kFineRounds; ++r) cnt += __popc(warp_transpose(m[r], lane));
        s_cw[warp][lane] = cnt;
        __syncthreads();
        if (warp == 0) {
            uint32_t sum = 0;
#pragma unroll
            for (int w = 0; w < kFineWarps; ++w) sum += s_cw[w][lane];
            wc[32ull * v + lane] = sum;  // 32 v + 31 < capacity
        }
        __syncthreads();
    }
}

// One CTA per super-tile: exclusive scan of its blocks' per-tile counts (in place), the tiles'
// pair counts stt[32 s + x] and the super-tile's pairs ssum[s].  The last CTA then scans the
// super-tiles' pairs into their first pair sbase[s], sets the pair count and scans the tile order's buckets.
__global__ void __launch_bounds__(256)
k_seg_scan(int64_t capacity, int TX, int TY, uint32_t* __restrict__ wc, Scratch sc,
           const RenderDesc* __restrict__ renders, int R) {
    pdl_begin();
    __shared__ uint32_t s_part[8][32];
    const int s = blockIdx.x, x = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t v0 = sc.vbase[s], nb = sc.vbase[s + 1] - v0;
    const uint32_t q = (nb + 7) / 8, r0 = min(nb, w * q), r1 = min(nb, r0 + q);
    uint32_t sum = 0;
    for (uint32_t r = r0; r < r1; ++r) {
        const uint64_t idx = 32ull * (v0 + r) + x;
        if (idx < (uint64_t)capacity) sum += wc[idx];
    }
    s_part[w][x] = sum;
    __syncthreads();
    uint32_t run = 0, total = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t p = s_part[k][x];
        run += k < w ? p : 0u;
        total += p;
    }
    for (uint32_t r = r0; r < r1; ++r) {
        const uint64_t idx = 32ull * (v0 + r) + x;
        if (idx < (uint64_t)capacity) {
            const uint32_t c = wc[idx];
            wc[idx] = run;
            run += c;
        }
    }
    if (w == 0) {
        sc.stt[32 * s + x] = total;
        const uint32_t all = __reduce_add_sync(kFull, total);
        if (x == 0) sc.ssum[s] = all;
        bucket_add(sc.tile_buckets, tile_of_bit(super_cell((uint32_t)s, TX, TY, renders, R), (uint32_t)x) >= 0, total);
    }
    if (!last_cta(&sc.bin_ticket[1])) return;
    if (w == 1) {  // tile_buckets: [0, 128) counts, zero again for the next render, [128, 256) cursors
        uint4* const counts = reinterpret_cast<uint4*>(sc.tile_buckets);
        static_assert(kOrderBuckets == 128, "four buckets a lane");
        const uint4 c = __ldcg(&counts[x]);
        uint32_t incl = c.x + c.y + c.z + c.w;
        const uint32_t own = incl;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, incl, o);
            if (x >= o) incl += t;
        }
        const uint32_t f = incl - own;
        counts[32 + x] = make_uint4(f, f + c.x, f + c.x + c.y, f + c.x + c.y + c.z);
        counts[x] = make_uint4(0u, 0u, 0u, 0u);
    }
    const unsigned long long P = cta_scan(
        (int)gridDim.x, [&](int k) { return (unsigned long long)__ldcg(&sc.ssum[k]); },
        [&](int k, unsigned long long v) { sc.sbase[k] = (uint32_t)v; });
    if (threadIdx.x == 0) {
        *sc.pair_count = P;
        if (P > *sc.pair_need) *sc.pair_need = P;
        if (P > (unsigned long long)capacity) atomicOr(sc.status, kStatusCapacity);
    }
}

// The pairs of every block (values = canonical indices into out), and the ranges of a super-tile's
// tiles from its first block.  Tile by tile, the warp's lanes whose entries reach it write side by side: an
// entry's pairs written by its own lane go to a line each, 32 different ones an instruction, and
// the lane with the most tiles holds its warp (39 us for the 6.5 M pairs of 500k Gaussians at
// 1920x1080, 27 us now; put together in shared memory first and written in runs of a block, 50 us).
__global__ void __launch_bounds__(kFineThreads)
k_fine_emit(int64_t capacity, int TX, int TY, const uint32_t* __restrict__ cv, const uint32_t* __restrict__ gidx,
            const uint32_t* __restrict__ gmask, const uint32_t* __restrict__ wc, int S, uint32_t tiles,
            uint32_t* __restrict__ out, Scratch sc, const RenderDesc* __restrict__ renders, int R) {
    pdl_begin();
    __shared__ uint32_t s_cw[kFineWarps * kFineRounds][32];
    __shared__ __align__(16) uint32_t s_off[kFineWarps * kFineRounds][32];  // of a warp's round, tile by tile
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t cap = capacity < 0xffffffffll ? (uint32_t)capacity : 0xffffffffu;
    const uint32_t VB = sc.vbase[S];
    for (uint32_t v = blockIdx.x; v < VB; v += gridDim.x) {
        if ((uint64_t)v >= (uint64_t)capacity / 32) break;
        const uint4 bi = sc.binfo[v];
        const uint32_t s = bi.x;
        uint32_t g[kFineRounds], m[kFineRounds];
#pragma unroll
        for (int r = 0; r < kFineRounds; ++r) {
            const uint64_t e = (uint64_t)bi.y + warp * (32 * kFineRounds) + r * 32 + lane;
            const bool valid = e < bi.z;
            const uint32_t e0 = valid ? cv[e] : 0u;
            g[r] = valid ? gidx[e0] : 0u;
            m[r] = valid ? gmask[e0] : 0u;
        }
#pragma unroll
        for (int r = 0; r < kFineRounds; ++r)  // lanes whose entry of round r reaches tile `lane`
            s_cw[warp * kFineRounds + r][lane] = __popc(warp_transpose(m[r], lane));
        __syncthreads();
        if (warp == 0) {
            const uint32_t tt = sc.stt[32 * s + lane];
            uint32_t incl = tt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += t;
            }
            const uint32_t ts = sc.sbase[s] + incl - tt;  // the tile's first pair
            uint32_t base = ts + wc[32ull * v + lane];
#pragma unroll
            for (int w = 0; w < kFineWarps * kFineRounds; ++w) {
                s_off[w][lane] = base;
                base += s_cw[w][lane];
            }
            if (bi.w == 0) {
                const int64_t tile = tile_of_bit(super_cell(s, TX, TY, renders, R), (uint32_t)lane);
                if (tile >= 0) sc.ranges[tile] = make_uint2(min(ts, cap), min(ts + tt, cap));
            }
        }
        __syncthreads();
#pragma unroll 2
        for (int x0 = 0; x0 < 32; x0 += 4)
#pragma unroll
            for (int r = 0; r < kFineRounds; ++r) {
                const uint4 off = *reinterpret_cast<const uint4*>(&s_off[warp * kFineRounds + r][x0]);
                const uint32_t at[4] = {off.x, off.y, off.z, off.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const bool in = (m[r] >> (x0 + k)) & 1u;
                    const uint32_t pos = at[k] + __popc(__ballot_sync(kFull, in) & lt);
                    if (in && pos < cap) out[pos] = g[r];
                }
            }
        __syncthreads();
    }
    // every super-tile's places in the compositing schedule, whether or not it has blocks
    if (warp == kFineWarps - 1)
        for (int s = blockIdx.x; s < S; s += gridDim.x) {
            const int64_t tile = tile_of_bit(super_cell((uint32_t)s, TX, TY, renders, R), (uint32_t)lane);
            const uint32_t pos = bucket_add(sc.tile_buckets + kOrderBuckets, tile >= 0, sc.stt[32 * s + lane]);
            if (tile >= 0 && pos < tiles) sc.tile_order[pos] = (uint32_t)tile;
            if (tile >= 0 && pos >= tiles) atomicOr(sc.status, kStatusInternal);
        }
}

// no entries at all (no capacity for any): the tiles in their own order
__global__ void k_tile_order_empty(int tiles, Scratch sc) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < tiles) sc.tile_order[t] = (uint32_t)t;
}

}  // namespace

// a pass reorders a whole CTA tile of keys in dynamic shared memory (32 KB with 4096 32-bit keys,
// 48 KB with 4096 64-bit keys)
template <typename KeyT, int kItems, int kThreads = kSortThreads>
void enable_scatter_smem() {
    static bool done = [] {
        cudaFuncSetAttribute(k_onesweep<KeyT, kItems, kThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)scatter_smem<KeyT, kItems, kThreads>());
        return true;
    }();
    (void)done;
}

// LSD passes over bits [first_shift, first_shift + bits) of the keys in keys[0] / keys[1] (viewed
// as KeyT), 8 bits a pass (the last pass takes what is left: bits above the range never take part),
// CTA tiles of kThreads x kItems keys: the digit totals of every pass in one read of the keys,
// then one launch per pass.  Returns the launches and leaves the sorted buffer's index in *out_buf.
// bits of a super-tile id (the coarse sort's key width)
static int super_bits(int64_t supers) {
    int bits = 0;
    while ((1ll << bits) < (long long)supers) ++bits;
    return bits;
}

// cleared: the look-back words (and, unless totals_ready, the digit totals) are already zero.  spare: there may be
// fewer keys than the capacity.
template <typename KeyT, int kItems, int kThreads = kSortThreads>
int sort_passes(int64_t capacity, int first_shift, int bits, const Scratch& sc, cudaStream_t s, int* out_buf,
                bool totals_ready = false, bool cleared = false, bool spare = true) {
    constexpr int kTile = kThreads * kItems;
    const int passes = (bits + kRadixBits - 1) / kRadixBits;
    const uint32_t last_mask = passes > 0 ? (uint32_t)((1u << (bits - kRadixBits * (passes - 1))) - 1u) : 0u;
    const int sb_max = (int)((capacity + kTile - 1) / kTile);
    // the totals read every key once: one CTA per 1024 keys, at most 8 per SM
    const int64_t want = (capacity + 1023) / 1024;
    const int total_blocks = (int)(want < 152 * 8 ? (want > 0 ? want : 1) : 152 * 8);
    int buf = 0;
    *out_buf = 0;
    if (sb_max <= 0 || passes <= 0) return 0;
    enable_scatter_smem<KeyT, kItems, kThreads>();
    KeyT* k[2] = {reinterpret_cast<KeyT*>(sc.keys[0]), reinterpret_cast<KeyT*>(sc.keys[1])};
    // abort word, tickets and the look-back words of every pass start cleared
    if (!cleared) cudaMemsetAsync(sc.sort_hist, 0, sizeof(uint32_t) * lookback_words(passes, sb_max), s);
    if (!totals_ready) {  // else the kernel that wrote the keys counted their digits
        if (!cleared) cudaMemsetAsync(sc.digit_totals, 0, sizeof(uint32_t) * kTotalWords, s);
        launch_pdl(k_digit_totals<KeyT>, dim3(total_blocks), dim3(kSortThreads), 0, s, capacity, first_shift, passes,
                   last_mask, (const KeyT*)k[0], sc);
    }
    for (int p = 0; p < passes; ++p) {
        const int shift = first_shift + p * kRadixBits;
        const uint32_t dmask = p == passes - 1 ? last_mask : (uint32_t)(kRadix - 1);
        launch_pdl(k_onesweep<KeyT, kItems, kThreads>, dim3(sb_max), dim3(kThreads), scatter_smem<KeyT, kItems, kThreads>(),
                   s, capacity, p, shift, dmask, sb_max, spare, (const KeyT*)k[buf], (const uint32_t*)sc.vals[buf], k[buf ^ 1],
                   sc.vals[buf ^ 1], sc);
        buf ^= 1;
    }
    *out_buf = buf;
    return (totals_ready ? 0 : 1) + passes;
}

// One radix-sort pass over three tiles of the pair buffers, the first never published: the ticket starts at
// 1, so tile 1 waits on tile 0 until its bound runs out (failure-detection self-test).
__global__ void k_selftest_setup(Scratch sc) {
    *sc.pair_count = 3ull * kSortTile;
    *sc.sort_blocks = 3u;
    sc.sort_hist[1] = 1u;  // the pass's ticket: tile 0 is never taken
}

int launch_timeout_selftest(int64_t capacity, const Scratch& sc, cudaStream_t s) {
    if (capacity < 3 * (int64_t)kSortTile) return 0;
    enable_scatter_smem<uint32_t, kSortItems>();
    const int sb_max = (int)((capacity + kSortTile - 1) / kSortTile);
    cudaMemsetAsync(sc.digit_totals, 0, sizeof(uint32_t) * kTotalWords, s);
    cudaMemsetAsync(sc.sort_hist, 0, sizeof(uint32_t) * lookback_words(1, sb_max), s);
    k_selftest_setup<<<1, 1, 0, s>>>(sc);
    uint32_t* k0 = reinterpret_cast<uint32_t*>(sc.keys[0]);
    uint32_t* k1 = reinterpret_cast<uint32_t*>(sc.keys[1]);
    k_onesweep<uint32_t, kSortItems><<<2, kSortThreads, scatter_smem<uint32_t, kSortItems>(), s>>>(
        capacity, 0, 0, kRadix - 1, sb_max, false, k0, sc.vals[0], k1, sc.vals[1], sc);
    return 2;
}

int launch_depth_sort(int64_t n, const Scratch& sc, cudaStream_t s, const uint32_t** perm, bool cleared) {
    Scratch d = sc;
    d.keys[0] = sc.dkeys[0];
    d.keys[1] = sc.dkeys[1];
    d.vals[0] = sc.dvals[0];
    d.vals[1] = sc.dvals[1];
    d.sort_hist = sc.dhist;
    d.digit_totals = sc.dtotals;
    d.pair_count = sc.dcount;
    d.sort_blocks = sc.dblocks;
    int buf = 0;
    const int launched = sort_passes<uint32_t, kDepthItems, kDepthThreads>(n, 0, 32, d, s, &buf, false, cleared, false);
    *perm = sc.dvals[buf];
    return launched;
}

int launch_bin_count(int64_t n, int64_t supers, int64_t capacity, const uint32_t* perm, const Scratch& sc,
                     cudaStream_t s, bool cleared) {
    const int64_t nbk = (n + kProjBlock - 1) / kProjBlock;
    const int nb = (int)((nbk + kCountItems - 1) / kCountItems);
    if (!cleared) cudaMemsetAsync(sc.pair_count, 0, sizeof(unsigned long long), s);
    launch_pdl(k_coarse_counts, dim3(nb > 0 ? nb : 1), dim3(kProjBlock), 0, s, n, capacity, supers, perm, sc);
    return 1;
}

int launch_bin_lists(int64_t n, int TX, int TY, int T, int64_t tiles, int64_t supers, int64_t capacity,
                     const uint32_t* perm, const Scratch& sc, cudaStream_t s, int* out_buf, const RenderDesc* renders,
                     int R, bool cleared) {
    const int nb = (int)((n + kProjBlock - 1) / kProjBlock);
    int launched = 0;
    *out_buf = 1;
    // canonical index and reach mask of coarse entry e0 in the upper halves of the key buffers (the
    // coarse keys are 32-bit: the sort uses the lower halves)
    uint32_t* gidx = reinterpret_cast<uint32_t*>(sc.keys[0]) + capacity;
    uint32_t* gmask = reinterpret_cast<uint32_t*>(sc.keys[1]) + capacity;
    if (!cleared) cudaMemsetAsync(sc.ranges, 0, sizeof(uint2) * (size_t)tiles, s);
    if (capacity <= 0 || supers <= 0) {
        if (tiles <= 0) return 0;
        k_tile_order_empty<<<(unsigned)((tiles + 255) / 256), 256, 0, s>>>((int)tiles, sc);
        return 1;
    }
    const int bits = super_bits(supers);
    const int passes = (bits + kRadixBits - 1) / kRadixBits;
    const uint32_t last_mask = passes > 0 ? (uint32_t)((1u << (bits - kRadixBits * (passes - 1))) - 1u) : 0u;
    if (!cleared) cudaMemsetAsync(sc.digit_totals, 0, sizeof(uint32_t) * kTotalWords, s);
    if (nb > 0) {
        const bool few = nb < 4 * 152;
        launch_pdl(few ? k_coarse_emit<4> : k_coarse_emit<1>, dim3(nb), dim3(kProjBlock * (few ? 4 : 1)), 0, s, n,
                   (TX + kSuperW - 1) / kSuperW, T, capacity, perm, sc, gidx, gmask, passes, last_mask, renders, R);
        ++launched;
    }
    // the coarse entries arrive in depth order: a stable sort by super-tile keeps it in each
    // super-tile (its count and CTA count are the coarse stage's, its digit totals the emission's)
    Scratch cs = sc;
    cs.pair_count = sc.coarse_count;
    int cb = 0;
    launched += sort_passes<uint32_t, kCoarseItems, kCoarseThreads>(capacity, 0, bits, cs, s, &cb, true, cleared);
    int crange_from = passes == 0 ? 2 : 1;
    if (passes > 1) {  // the super-tiles' ranges from the sorted keys
        if (!cleared) cudaMemsetAsync(sc.crange, 0, sizeof(uint2) * (size_t)supers, s);
        cs.ranges = sc.crange;
        launch_pdl(k_ranges, dim3(152 * 8), dim3(256), 0, s, capacity, (uint32_t)supers,
                   reinterpret_cast<const uint32_t*>(sc.keys[cb]), cs);
        ++launched;
        crange_from = 0;
    }
    launch_pdl(k_block_prefix, dim3(1), dim3(kScanThreads), 0, s, (int)supers, capacity, sc, crange_from);
    // block counts over the sorted coarse keys (read by k_ranges before)
    uint32_t* wc = reinterpret_cast<uint32_t*>(sc.keys[cb]);
    const uint32_t* cv = sc.vals[cb];
    launch_pdl(k_fine_count, dim3(kFineGrid), dim3(kFineThreads), 0, s, capacity, cv, gmask, wc, (int)supers, sc);
    launch_pdl(k_seg_scan, dim3((unsigned)supers), dim3(256), 0, s, capacity, TX, TY, wc, sc, renders, R);
    launch_pdl(k_fine_emit, dim3(kFineGrid), dim3(kFineThreads), 0, s, capacity, TX, TY, cv, gidx, gmask, wc, (int)supers,
               (uint32_t)tiles, sc.vals[cb ^ 1], sc, renders, R);
    *out_buf = cb ^ 1;
    return launched + 4;
}

ZeroPlan render_zero_plan(const Scratch& sc, int64_t n, int64_t tiles, int64_t supers, int64_t capacity) {
    ZeroPlan z{};
    auto add = [&](void* p, size_t words) {
        if (p && words > 0 && z.count < kZeroRegions) {
            z.p[z.count] = static_cast<uint32_t*>(p);
            z.words[z.count] = (uint32_t)words;
            ++z.count;
        }
    };
    // depth sort: 4 passes over ceil(n / kDepthTile) tiles, its digit totals
    add(sc.dhist, lookback_words(32 / kRadixBits, (n + kDepthTile - 1) / kDepthTile));
    add(sc.dtotals, kTotalWords);
    add(sc.pair_count, 2);
    add(sc.ranges, 2 * (size_t)tiles);
    // coarse stage: its digit totals, its sort's look-back words, the super-tiles' ranges
    add(sc.digit_totals, kTotalWords);
    if (capacity > 0 && supers > 0) {
        const int passes = (super_bits(supers) + kRadixBits - 1) / kRadixBits;
        add(sc.sort_hist, lookback_words(passes, (capacity + kSortTile - 1) / kSortTile));
        if (passes > 1) add(sc.crange, 2 * (size_t)supers);
    }
    add(sc.l1_acc, 6);  // the forward's fused L1 sums and ticket
    return z;
}

void clear_zero_plan(const ZeroPlan& z, cudaStream_t s) {
    for (int r = 0; r < z.count; ++r) cudaMemsetAsync(z.p[r], 0, sizeof(uint32_t) * z.words[r], s);
}

int launch_radix_sort_only(int64_t capacity, int key_bits, const Scratch& sc, cudaStream_t s,
                           int* out_buf) {
    return sort_passes<unsigned long long, kSortItems>(capacity, 0, key_bits, sc, s, out_buf);
}

}  // namespace pgs
