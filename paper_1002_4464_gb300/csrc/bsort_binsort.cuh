// bsort_binsort.cuh -- one-pass distribution sort of the keys held by one
// CTA (Step 2, Step 9 and whole units of GPU Bucket Sort, Dehne & Zaboli,
// Section 4, Algorithm 1, which may use any exact sort).
//
// Equal keys of a keys-only sort are indistinguishable, so nothing has to be
// stable, and one counting pass over many bins replaces the digit passes (or
// merge levels): the NB bins cut the unit's key range [kmin, kmax] linearly
// (float keys: their values), about one key per bin;
//   1. every key adds one to its bin's 16-bit counter (shared-memory
//      reductions; two bins per word: bin b is the low half of word b for
//      b < NB/2, the high half of word b - NB/2 otherwise);
//   2. one exclusive scan of the counters, and the largest bin's count G;
//   3. an atomic add on its bin's counter gives each key its rank, where it
//      is stored;
//   4. the keys are now sorted by bin, so every key is within G of its place:
//      each thread reloads E consecutive keys and G phases of odd-even
//      transposition (one min and one max per pair, neighbouring lanes by
//      shuffles) order them.  Groups of one bin that straddle two warps are
//      merged afterwards, 32 keys either side.
// What bounds it: the shared-memory pipe (49 % busy in 32768-key units, DRAM
// 24 %, 58 instructions a key; a random-bank atomic takes about six wavefronts
// per warp, the scatter three) and the barriers between the steps with one or
// two CTAs per SM.  2^26 keys on a GB300, load and store included, before the
// sample of crowding (1 % more with it): as 32768-key units 255 us (512 threads x 64 keys; five
// 7-bit digit passes took 513 us, for 19 varying bits three passes 338 us),
// as 16384-key units 203 us (two CTAs of 512 x 32 per SM; comparison sort
// 588 us), 8192: 189 us (448), 4096: 191 us (369), 2048: 174 us (314).  1024
// threads x 32 keys for 32768 keys measured 283 us (64 registers spill).
// 2^25 64-bit keys, pairs in brackets: as 16384-item units 240 us (224;
// comparison sort 771 and 776), 8192: 201 (190; 707), 4096: 176 (160; 519),
// 2048: 158 (137; 524).
// A range below NB gives every value a bin of its own (several, when there
// are fewer values than lanes, so that a warp's atomics do not meet on one
// counter) and needs no step 4.
//
// Keys that crowd.  Before anything is counted, one key of each thread is
// sampled and its place in the map's bins is looked at (BinSort::crowding);
// where they meet far more often than a smooth density's do, the unit takes
//   the bins of the logarithm of key - kmin (bin_again; floats: of their
//   codes), if the sample is spread there: keys over many scales, or most of
//   them near kmin and some far off;
//   the same bins, if the sample says that cutting each of them once more, as
//   below, parts the keys: a few smooth groups;
//   else the sort that the bins replaced (bin_other): comparisons, digits for
//   32768-key units of 32-bit keys, merges where the unit is made of runs.
// A unit that passes may still have a bin of more than kBinPhases keys: a value
// repeated often, or two that share a bin.  bin_skewed then cuts every bin b
// of n_b keys once more, linearly into n_b bins at positions [P_b, P_b + n_b)
// of the order, so that crowded stretches of the range get as many bins as
// they hold keys.  (A bin with an eighth of the unit or more takes every 16th
// of those positions, and its keys are spread over the 16 by lane: a value
// repeated that often would otherwise meet on one counter; pairs, whose equal
// keys must keep their order, are instead cut a third time, by position.)
// Where the sample sent the unit here, it is looked at again in the refined
// bins.  What is left unordered
// inside them is put right by up to kBinPhases phases, by a comparison sort
// of the warps where that is not enough, and by bin_other when two warps still
// overlap.
// Batches of 2^26 32-bit (2^25 64-bit) keys as units of 32768 (16384): even
// keys 350 us (296); 1024 values, Zipf 1.1, 564 (400); keys spread over their
// logarithm 575 (484), one far key to a unit 574 (496), 50 narrow groups 682
// (907); all of these took 655 (835) by digits (comparisons) alone.  As units
// of 2048: 674 (414); 850 (545), 845 (600), 849 (554), 849 (821) against 835
// (795).
#pragma once

#include <cstdint>

#include "bsort_device.cuh"
#include "bsort_radix.cuh"

namespace bsort {

constexpr uint32_t kBinPhases = 32;  // largest bin ordered by phases alone

// Bins of a unit of T*E keys.
template <typename K, int T, int E>
constexpr int bin_count() { return T * E; }

// Shared memory of cta_bin_sort: the keys in the padded layout, then NB
// 16-bit counters (16-byte aligned) and a spare word per lane; at least what
// the digit sort of crowded units takes.
template <typename K, int T, int E>
struct BinSmem {
    static constexpr int kKeyBytes = (padded_elems<K>(T * E) * (int)sizeof(K) + 15) & ~15;
    static constexpr int kBins = kKeyBytes + bin_count<K, T, E>() * 2 + 32 * 4;
    static constexpr int digits()
    {
        if constexpr (sizeof(K) == 4 && T * E == 32768) return RadixSmem<T, E, 6>::kBytes;
        else return 0;
    }
    static constexpr int kBytes = kBins > digits() ? kBins : digits();
};

// One phase pair (even, then odd positions) of odd-even transposition over
// the warp's 32*E keys in blocked order.
template <typename K, int E>
__device__ __forceinline__ void transpose_phases(K (&v)[E], int lane)
{
#pragma unroll
    for (int k = 0; k + 1 < E; k += 2) cmp_swap(v[k], v[k + 1]);
#pragma unroll
    for (int k = 1; k + 1 < E; k += 2) cmp_swap(v[k], v[k + 1]);
    const K x = __shfl_down_sync(0xFFFFFFFFu, v[0], 1);
    const K y = __shfl_up_sync(0xFFFFFFFFu, v[E - 1], 1);
    if (lane < 31) v[E - 1] = kmin<K>(v[E - 1], x);
    if (lane > 0) v[0] = kmax<K>(v[0], y);
}

// Whether the warp's keys (blocked order) still hold an inversion.
template <typename K, int E>
__device__ __forceinline__ bool warp_inverted(const K (&v)[E], int lane)
{
    bool bad = false;
#pragma unroll
    for (int k = 0; k + 1 < E; ++k) bad |= v[k] > v[k + 1];
    const K x = __shfl_down_sync(0xFFFFFFFFu, v[0], 1);
    bad |= lane < 31 && v[E - 1] > x;
    return __any_sync(0xFFFFFFFFu, bad) != 0;
}

// Monotone maps of a unit's keys, kmin = lo < kmax = hi, to bins [0, NB):
// bin(key), and fine(key) = the key's place inside its bin as a 32-bit
// fraction.
//
// By key value.
template <typename K, int NB> struct BinMap;

// The largest multiplier, or a few less, with d * mult < NB * 2^32, for d >=
// 2^31: every thread works it out, and a 64-bit division would take a tenth
// of a small unit's time.  The quotient lies in (NB, 2 NB]; its rounding up
// by 2^-21 at most is taken off before the fraction is.
template <int NB>
__device__ __forceinline__ uint32_t bin_mult(uint32_t d)
{
    return __float2uint_rz(__fdividef((float)NB * 4294967296.0f, __uint2float_ru(d)) *
                           (1.0f - 1.0f / (1 << 20)));
}

template <int NB> struct BinMap<uint32_t, NB> {
    uint32_t base, mult;
    int lz;
    __device__ BinMap(uint32_t lo, uint32_t hi)
    {
        base = lo;
        lz = __clz((int)(hi - lo));
        mult = bin_mult<NB>((hi - lo) << lz);
    }
    __device__ uint32_t bin(uint32_t key) const { return __umulhi((key - base) << lz, mult); }
    __device__ uint32_t fine(uint32_t key) const { return ((key - base) << lz) * mult; }
};

template <int NB> struct BinMap<uint64_t, NB> {
    uint64_t base;
    uint32_t mult;
    int sr, sl;  // the top 32 bits of key - base: >> sr, then << sl
    __device__ BinMap(uint64_t lo, uint64_t hi)
    {
        base = lo;
        const int z = __clzll((long long)(hi - lo));
        sr = z < 32 ? 32 - z : 0;
        sl = z < 32 ? 0 : z - 32;
        mult = bin_mult<NB>(top(hi));
    }
    __device__ uint32_t top(uint64_t key) const { return (uint32_t)((key - base) >> sr) << sl; }
    __device__ uint32_t bin(uint64_t key) const { return __umulhi(top(key), mult); }
    __device__ uint32_t fine(uint64_t key) const { return top(key) * mult; }
};

// Codes of floats by float value: equal-width bins of [fmin, fmax].  The
// difference, the product and the rounding to 2^-23 of the range are each
// monotone, so the map is.
template <int NB> struct BinMapF32 {
    float lo, scale;
    bool ok;
    __device__ BinMapF32(uint32_t lo_code, uint32_t hi_code)
    {
        lo = __uint_as_float(f32_decode(lo_code));
        const float d = __uint_as_float(f32_decode(hi_code)) - lo;
        // (the margin keeps the rounded product inside [0, 2^23))
        scale = 8388600.0f / d;
        ok = d > 0.0f && d < 3.0e38f && scale > 0.0f && scale < 3.0e38f;  // false with NaN, inf
    }
    __device__ uint32_t place(uint32_t key) const  // 2^23 + place, as float bits
    {
        return __float_as_uint(
            fmaf(__uint_as_float(f32_decode(key)) - lo, scale, 8388608.0f));
    }
    static constexpr int kShift = 23 - __builtin_ctz(NB);
    __device__ uint32_t bin(uint32_t key) const { return (place(key) >> kShift) & (uint32_t)(NB - 1); }
    // (2^kShift places a bin, 256 of a 32768-key unit: a bin of more keys is cut
    // at no more.  What the rounding left, an fma away, would add bits; it
    // made units of 1024 repeated values 8 % slower and helps few)
    __device__ uint32_t fine(uint32_t key) const { return place(key) << (32 - kShift); }
};

// Pairs (key << 32 | position) by key.
template <int NB> struct BinMapPairs {
    BinMap<uint32_t, NB> m;
    __device__ BinMapPairs(uint32_t lo, uint32_t hi) : m(lo, hi) {}
    __device__ uint32_t bin(uint64_t x) const { return m.bin((uint32_t)(x >> 32)); }
    __device__ uint32_t fine(uint64_t x) const { return m.fine((uint32_t)(x >> 32)); }
};

// By the logarithm of key - kmin, as its rounded-down float's code has it:
// keys spread over their logarithm, or crowded near kmin with others far off.
template <typename K, int NB> struct BinMapLog {
    K base;
    BinMap<uint32_t, NB> m;
    __device__ BinMapLog(K lo, K hi) : base(lo), m(0u, code(hi - lo)) {}
    static __device__ uint32_t code(K x)  // 0, then from 1's code on
    {
        float f;
        if constexpr (sizeof(K) == 4) f = __uint2float_rz(x);
        else f = __ull2float_rz(x);
        return x == 0 ? 0u : __float_as_uint(f) - 0x3F000000u;
    }
    __device__ uint32_t bin(K key) const { return m.bin(code(key - base)); }
    __device__ uint32_t fine(K key) const { return m.fine(code(key - base)); }
};
template <int NB> struct BinMapLogPairs {
    BinMapLog<uint32_t, NB> m;
    __device__ BinMapLogPairs(uint32_t lo, uint32_t hi) : m(lo, hi) {}
    __device__ uint32_t bin(uint64_t x) const { return m.bin((uint32_t)(x >> 32)); }
    __device__ uint32_t fine(uint64_t x) const { return m.fine((uint32_t)(x >> 32)); }
};

// Ranges below NB: value x of the range has the rep bins [x*rep, (x+1)*rep),
// a power of two up to 32, spread over the lanes.
template <typename K, int NB> struct BinMapExact {
    K base;
    int shift;
    uint32_t off;
    __device__ BinMapExact(K lo, K hi, int lane)
    {
        base = lo;
        const uint32_t per = (uint32_t)NB / ((uint32_t)(hi - lo) + 1u);  // >= 1
        shift = min(31 - __clz((int)per), 5);
        off = (uint32_t)lane & ((1u << shift) - 1u);
    }
    __device__ uint32_t bin(K key) const { return ((uint32_t)(key - base) << shift) + off; }
};

// The shape of one CTA's bin sort and its steps.
template <typename K, int T, int E>
struct BinSort {
    static constexpr int NB = bin_count<K, T, E>();
    static constexpr int CAP = T * E;
    static constexpr int W = 32 * E;      // keys of a warp
    static constexpr int NWARP = T / 32;
    static constexpr int NW = NB / 2;     // counter words
    static constexpr int IT = NW / NWARP / 128;  // 16-byte words a lane scans
    static_assert(T % 32 == 0 && T >= 64 && T <= 1024 && E % 8 == 0, "whole warps");
    static_assert((NB & (NB - 1)) == 0 && NB <= 32768 && IT >= 1, "power-of-two bins, whole words");
    static_assert(CAP <= 32768, "counts and ranks fit 16 bits");

    K *sm;
    int len, tid, lane, warp;
    bool full, act;  // the warp holds no padding / any real key
    uint32_t cbase;  // shared address of the counters

    __device__ BinSort(K *sm_, int len_) : sm(sm_), len(len_)
    {
        tid = (int)threadIdx.x;
        lane = tid & 31;
        warp = tid >> 5;
        full = (warp + 1) * W <= len;
        act = warp * W < len;
        cbase = smem_u32addr(sm) + (uint32_t)BinSmem<K, T, E>::kKeyBytes;
    }
    // shared address of bin b's counter word and the bin's half
    __device__ uint32_t word(uint32_t b) const { return cbase + ((b & (uint32_t)(NW - 1)) << 2); }
    static __device__ uint32_t half(uint32_t b) { return (b / (uint32_t)NW) << 4; }
    __device__ bool real(int k) const { return wb_pos<E>(warp, lane, k) < len; }
    __device__ uint32_t spare() const { return cbase + 4u * (uint32_t)(NW + lane); }
    __device__ uint4 *counters() const
    {
        return reinterpret_cast<uint4 *>(reinterpret_cast<unsigned char *>(sm) +
                                         BinSmem<K, T, E>::kKeyBytes);
    }

    template <bool FULL, typename F>
    __device__ __forceinline__ void count(const K (&v)[E], const F &map) const
    {
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const uint32_t b = map.bin(v[k]);
            red_add_shared(FULL || real(k) ? word(b) : spare(), 1u << half(b));
        }
    }
    // Exclusive scan of the counters at `in` (NB of them) into `out`, in bin
    // order; returns the largest count.  s_a, s_b: a word per warp.
    __device__ __forceinline__ uint32_t scan(const uint4 *in, uint4 *out, uint32_t *s_a,
                                             uint32_t *s_b) const
    {
        // warp w scans words [w*NW/NWARP, (w+1)*NW/NWARP), 128 at a time
        const int at = warp * (NW / NWARP / 4) + lane;
        uint32_t gm = 0, s = 0;
#pragma unroll 2  // (the keys stay live in registers)
        for (int i = 0; i < IT; ++i) {
            const uint4 c = in[at + i * 32];
            gm = __vmaxu2(gm, __vmaxu2(__vmaxu2(c.x, c.y), __vmaxu2(c.z, c.w)));
            s += c.x + c.y + c.z + c.w;
        }
        s = __reduce_add_sync(0xFFFFFFFFu, s);
        gm = __reduce_max_sync(0xFFFFFFFFu, max(gm & 0xFFFFu, gm >> 16));
        if (lane == 0) {
            s_a[warp] = s;
            s_b[warp] = gm;
        }
        __syncthreads();
        uint32_t inc = lane < NWARP ? s_a[lane % NWARP] : 0u;
        const uint32_t own = inc;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, inc, 31);
        uint32_t run = __shfl_sync(0xFFFFFFFFu, inc - own, warp);
        const uint32_t G = __reduce_max_sync(0xFFFFFFFFu, s_b[lane % NWARP]);
        run += (total & 0xFFFFu) << 16;  // high-half bins follow every low-half one
#pragma unroll 1
        for (int i = 0; i < IT; ++i) {
            const uint4 c = in[at + i * 32];
            const uint32_t sum = c.x + c.y + c.z + c.w;
            inc = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
                if (lane >= d) inc += y;
            }
            uint4 o;
            o.x = run + inc - sum;
            o.y = o.x + c.x;
            o.z = o.y + c.y;
            o.w = o.z + c.z;
            out[at + i * 32] = o;
            run += __shfl_sync(0xFFFFFFFFu, inc, 31);
        }
        __syncthreads();
        return G;
    }
    template <bool FULL, typename F>
    __device__ __forceinline__ void scatter(const K (&v)[E], const F &map) const
    {
        constexpr int GB = 4;  // atomics in flight per batch
#pragma unroll
        for (int k0 = 0; k0 < E; k0 += GB) {
            uint32_t r[GB];
#pragma unroll
            for (int j = 0; j < GB; ++j) {
                const uint32_t b = map.bin(v[k0 + j]);
                const uint32_t a = FULL || real(k0 + j) ? word(b) : spare();
                // (a rank is below CAP; the mask keeps every store inside
                // the key area whatever the counters hold)
                r[j] = (atom_add_shared(a, 1u << half(b)) >> half(b)) & (uint32_t)(CAP - 1);
            }
#pragma unroll
            for (int j = 0; j < GB; ++j)
                if (FULL || real(k0 + j)) sm[pidx<K>((int)r[j])] = v[k0 + j];
        }
    }
    // One of each thread's keys is sampled: register sample_reg(), which
    // differs between neighbouring lanes and between warps (units made of
    // sorted runs repeat their ranks from warp to warp).
    __device__ __forceinline__ int sample_at() const { return (lane + warp) & 7; }
    __device__ __forceinline__ int sample_reg() const { return sample_at() * (E / 8); }
    template <typename V>
    __device__ __forceinline__ V pick(const V (&a)[8]) const
    {
        const int i = sample_at();
        const V b = i & 1 ? a[1] : a[0], c = i & 1 ? a[3] : a[2];
        const V d = i & 1 ? a[5] : a[4], e = i & 1 ? a[7] : a[6];
        const V f = i & 2 ? c : b, g = i & 2 ? e : d;
        return i & 4 ? g : f;
    }
    __device__ __forceinline__ K sample(const K (&v)[E]) const
    {
        const K a[8] = {v[0],         v[E / 8],     v[2 * E / 8], v[3 * E / 8],
                        v[4 * E / 8], v[5 * E / 8], v[6 * E / 8], v[7 * E / 8]};
        return pick(a);
    }
    // Whether the sampled keys meet in bins more often than keys of a smooth
    // density do: each leaves its value at its bin's place in the key area (any
    // may stay), and those that find another one there are counted (ANY: those
    // that another thread's key replaced).  With S samples a density of rho
    // times the even one counts about S^2 rho / (2 NB) of them; the result is
    // their number over the one where rho is 16 (even keys: 1; a bell: 2.5; an
    // exponential: 5), so that above 1 the bins are crowded.  The key area is
    // overwritten; ends with a barrier.
    template <bool ANY, typename V>
    __device__ __forceinline__ float crowding(uint32_t bin, V value) const
    {
        const bool r = real(sample_reg());
        const V mark = ANY ? (V)tid : value;
        V *at = reinterpret_cast<V *>(sm) + (bin & (uint32_t)(CAP - 1));
        if (r) *at = mark;
        __syncthreads();
        const bool meets = r && *at != mark;
        const float fill = (float)len * (1.0f / CAP);
        constexpr float limit = T * (E >= 64 ? 0.115f : E >= 32 ? 0.213f : 0.368f);
        return __fdividef((float)__syncthreads_count(meets) - 4.0f, limit * fill * fill);
    }
    // Whether they would still do so with every bin cut once more (bin_skewed):
    // a sampled key whose bin holds c of them falls to place fine * c * E of
    // it; the pairs (bin, place) are looked at by a hash.  Ends with a barrier.
    template <typename V>
    __device__ __forceinline__ float crowding_cut(uint32_t bin, uint32_t fine, V value) const
    {
        uint32_t *at = reinterpret_cast<uint32_t *>(sm) + (bin & (uint32_t)(CAP - 1));
        const bool r = real(sample_reg());
        if (r) *at = 0u;
        __syncthreads();
        if (r) atomicAdd(at, 1u);
        __syncthreads();
        const uint32_t c = r ? *at : 0u;
        const uint32_t place = __umulhi(fine, c * (uint32_t)E);
        // (where an eighth of a large unit is in one bin they would queue for
        // its counter: as if crowded)
        if (__syncthreads_or(T >= 512 && c * 8u > (uint32_t)T)) return 2.0f;
        const uint32_t h = (bin * 0x9E3779B1u + place) * 0x85EBCA6Bu;
        return crowding<false>(h >> (32 - __builtin_ctz(CAP)), value);
    }
    // Bins that straddle this warp's first key: merge the last 32 keys before
    // it and the first 32 from it, each ascending.
    __device__ __forceinline__ void merge_edge() const
    {
        if (warp == 0 || !act) return;
        const int b = warp * W;
        const K x = sm[pidx<K>(b - 32 + lane)], y = sm[pidx<K>(b + 31 - lane)];
        K l = kmin<K>(x, y), h = kmax<K>(x, y);
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) {
            const K xl = __shfl_xor_sync(0xFFFFFFFFu, l, d);
            const K xh = __shfl_xor_sync(0xFFFFFFFFu, h, d);
            const bool low = (lane & d) == 0;
            l = low ? kmin<K>(l, xl) : kmax<K>(l, xl);
            h = low ? kmin<K>(h, xh) : kmax<K>(h, xh);
        }
        sm[pidx<K>(b - 32 + lane)] = l;
        sm[pidx<K>(b + lane)] = h;
    }
    // Step 4: order the keys inside the bins, at most G <= 32 keys each.
    __device__ __forceinline__ void order_bins(K (&v)[E], uint32_t G) const
    {
        if (act) {
#pragma unroll
            for (int k = 0; k < E; ++k) v[k] = sm[pidx<K>(tid * E + k)];
#pragma unroll 1
            for (uint32_t p = 0; p < G; p += 2) transpose_phases<K, E>(v, lane);
#pragma unroll
            for (int k = 0; k < E; ++k) sm[pidx<K>(tid * E + k)] = v[k];
        }
        __syncthreads();
        merge_edge();
        __syncthreads();
    }
    __device__ __forceinline__ void pad() const  // the positions behind the real keys
    {
        for (int x = len + tid; x < CAP; x += T) sm[pidx<K>(x)] = KeyMax<K>::v;
    }
};

// Sort of a unit that bins do not part: by digits or comparisons, or (run > 0)
// by merging its ascending runs of run keys.  The keys are in sm at their
// warp-blocked positions.  (This and bin_skewed are out of line, each by
// itself: their registers must not weigh on the usual path, nor on each other.)
template <typename K, int T, int E, bool RUNS>
__device__ __noinline__ void bin_other(K *sm, int len, int run)
{
    constexpr int CAP = T * E;
    const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
    K v[E];
    if constexpr (RUNS) {
        if (run >= 32 * E && run < CAP) {
#pragma unroll
            for (int k = 0; k < E; ++k) v[k] = sm[pidx<K>(k * T + tid)];
            __syncthreads();
#pragma unroll
            for (int k = 0; k < E; ++k) {  // odd runs descending, as the merges read them
                const int x = k * T + tid, q = x / run, o = x % run;
                sm[pidx<K>(q & 1 ? q * run + run - 1 - o : x)] = v[k];
            }
            __syncthreads();
            cta_merge_runs<K, T, E>(sm, run);
            return;
        }
    }
#pragma unroll
    for (int k = 0; k < E; ++k) v[k] = sm[pidx<K>(wb_pos<E>(warp, lane, k))];
    __syncthreads();
    if constexpr (sizeof(K) == 4 && CAP == 32768) cta_radix_sort<T, E, 6>(v, sm, len);
    else cta_sort<K, T, E>(v, sm, len);
}

// Sort of a unit whose first bins hold too many keys: each bin is cut once
// more.  The keys are in sm at their warp-blocked positions, the first bins'
// exclusive prefix P in the counters.  repeated: a bin that holds much of the
// unit does so by a repeated value.  False: the unit is not sorted, its keys
// are in sm in some order.
template <typename K, int T, int E, bool PAIRS, typename F>
__device__ __noinline__ bool bin_skewed(K *sm, int len, const F map, bool repeated)
{
    using B = BinSort<K, T, E>;
    constexpr int CAP = B::CAP, W = B::W, NWARP = B::NWARP, NW = B::NW;
    static_assert(B::NB == CAP, "the refined bins are positions of the order");
    static_assert(CAP * 2 <= BinSmem<K, T, E>::kKeyBytes, "their counters fit the key area");
    __shared__ uint32_t s_a[NWARP], s_b[NWARP];
    const B s(sm, len);
    const int tid = s.tid, lane = s.lane, warp = s.warp;
    // the sort key of an item (of a pair, without its position)
    auto value = [](K x) {
        if constexpr (PAIRS) return (uint32_t)(x >> 32);
        else return x;
    };
    K v[E];
#pragma unroll
    for (int k = 0; k < E; ++k) v[k] = sm[pidx<K>(wb_pos<E>(warp, lane, k))];
    __syncthreads();
    uint32_t *fine = reinterpret_cast<uint32_t *>(sm);  // the refined bins' counters
    const uint32_t *P = reinterpret_cast<const uint32_t *>(s.counters());
    const uint32_t fbase = smem_u32addr(fine);
    uint32_t bins[E / 2];  // the keys' bins so far, two to a word
    // Cut every bin by the keys' places in it (BY_POS: by their positions in
    // the unit, for pairs, whose equal keys keep their order).
    auto recount = [&](auto full, auto by_pos) {
        constexpr bool FULL = decltype(full)::value, BY_POS = decltype(by_pos)::value;
        constexpr int GB = 8;
#pragma unroll
        for (int k0 = 0; k0 < E; k0 += GB) {
            uint32_t p0[GB], p1[GB];
#pragma unroll
            for (int j = 0; j < GB; ++j) {
                const int k = k0 + j;
                const uint32_t b = BY_POS ? (bins[k / 2] >> (16 * (k & 1))) & 0xFFFFu
                                          : map.bin(v[k]) & (uint32_t)(B::NB - 1);
                const uint32_t e = b + 1;
                p0[j] = (P[b & (uint32_t)(NW - 1)] >> B::half(b)) & 0xFFFFu;
                p1[j] = e < (uint32_t)B::NB ? (P[e & (uint32_t)(NW - 1)] >> B::half(e)) & 0xFFFFu
                                            : (uint32_t)len;
            }
#pragma unroll
            for (int j = 0; j < GB; ++j) {
                const int k = k0 + j;
                const uint32_t w = p1[j] - p0[j];
                uint32_t at;
                if constexpr (BY_POS) {
                    at = w * (uint32_t)wb_pos<E>(warp, lane, k) / (uint32_t)CAP;
                } else {
                    const int sh = !PAIRS && repeated && w >= (uint32_t)(CAP / 8) ? 4 : 0;
                    at = (__umulhi(map.fine(v[k]), w >> sh) << sh) +
                         ((uint32_t)lane & ((1u << sh) - 1u));
                }
                const uint32_t b2 = (p0[j] + at) & (uint32_t)(CAP - 1);
                if constexpr (BY_POS)
                    bins[k / 2] = (bins[k / 2] & (0xFFFFu << (16 * (1 - (k & 1))))) |
                                  (b2 << (16 * (k & 1)));
                else if (k & 1) bins[k / 2] |= b2 << 16;
                else bins[k / 2] = b2;
                red_add_shared(FULL || s.real(k) ? fbase + ((b2 & (uint32_t)(NW - 1)) << 2)
                                                 : s.spare(),
                               1u << B::half(b2));
            }
        }
    };
    auto refine = [&](auto by_pos) {
        for (int i = tid; i < CAP / 8; i += T)
            reinterpret_cast<uint4 *>(fine)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        if (s.full) recount(std::true_type{}, by_pos);
        else if (s.act) recount(std::false_type{}, by_pos);
        __syncthreads();
        s.scan(reinterpret_cast<const uint4 *>(fine), s.counters(), s_a, s_b);
    };
    auto place = [&](auto full) {
        constexpr int GB = 8;
#pragma unroll
        for (int k0 = 0; k0 < E; k0 += GB) {
            uint32_t r[GB];
#pragma unroll
            for (int j = 0; j < GB; ++j) {
                const int k = k0 + j;
                const uint32_t b = (bins[k / 2] >> (16 * (k & 1))) & 0xFFFFu;
                const uint32_t a = decltype(full)::value || s.real(k) ? s.word(b) : s.spare();
                r[j] = (atom_add_shared(a, 1u << B::half(b)) >> B::half(b)) & (uint32_t)(CAP - 1);
            }
#pragma unroll
            for (int j = 0; j < GB; ++j)
                if (decltype(full)::value || s.real(k0 + j)) sm[pidx<K>((int)r[j])] = v[k0 + j];
        }
    };
    refine(std::false_type{});
    // keys of several scales crowd the refined bins too
    uint32_t a[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int k = j * (E / 8);
        a[j] = (bins[k / 2] >> (16 * (k & 1))) & 0xFFFFu;
    }
    if (!repeated && s.template crowding<false>(s.pick(a), value(s.sample(v))) > 1.0f) {
#pragma unroll
        for (int k = 0; k < E; ++k) sm[pidx<K>(wb_pos<E>(warp, lane, k))] = v[k];
        __syncthreads();
        return false;
    }
    if constexpr (PAIRS) refine(std::true_type{});
    if (s.full) place(std::true_type{});
    else if (s.act) place(std::false_type{});
    s.pad();
    __syncthreads();
#pragma unroll
    for (int k = 0; k < E; ++k) v[k] = sm[pidx<K>(tid * E + k)];
    if (s.act) {
        bool bad = warp_inverted<K, E>(v, lane);
#pragma unroll 1
        for (uint32_t p = 0; bad && p < kBinPhases; p += 8) {
#pragma unroll 1
            for (int q = 0; q < 4; ++q) transpose_phases<K, E>(v, lane);
            bad = warp_inverted<K, E>(v, lane);
        }
        if (bad) {
            sort_network<E>(v);
            warp_merge_levels<K, E>(v, lane);
        }
#pragma unroll
        for (int k = 0; k < E; ++k) sm[pidx<K>(tid * E + k)] = v[k];
    }
    __syncthreads();
    s.merge_edge();
    __syncthreads();
    const int b = warp * W;  // (false when two warps overlap by more)
    return !__syncthreads_or(warp > 0 && s.act &&
                             (sm[pidx<K>(b - 33)] > sm[pidx<K>(b - 32)] ||
                              sm[pidx<K>(b + 31)] > sm[pidx<K>(b + 32)]));
}

// The sort by the bins of another map, for units that crowd in the first one:
// the keys in sm at their warp-blocked positions, the counters zero.
template <typename K, int T, int E, bool PAIRS, typename F>
__device__ __noinline__ void bin_again(K *sm, int len, const F map)
{
    using B = BinSort<K, T, E>;
    __shared__ uint32_t s_a[B::NWARP], s_b[B::NWARP];
    const B s(sm, len);
    K v[E];
#pragma unroll
    for (int k = 0; k < E; ++k) v[k] = sm[pidx<K>(wb_pos<E>(s.warp, s.lane, k))];
    if (s.full) s.template count<true>(v, map);
    else if (s.act) s.template count<false>(v, map);
    __syncthreads();
    const uint32_t G = s.scan(s.counters(), s.counters(), s_a, s_b);
    if (G > kBinPhases) {
        if (!bin_skewed<K, T, E, PAIRS>(sm, len, map, true)) bin_other<K, T, E, false>(sm, len, 0);
        return;
    }
    if (s.full) s.template scatter<true>(v, map);
    else if (s.act) s.template scatter<false>(v, map);
    s.pad();
    __syncthreads();
    s.order_bins(v, G);
}

// Sort the CTA's T*E keys v ascending into sm (padded layout pidx, then the
// counters: BinSmem<K, T, E>::kBytes in all).  On entry v holds the keys in
// the warp-blocked layout; positions >= len are padding holding the maximal
// key.  On return sm[pidx(x)] is the x-th smallest key, padding after the
// len real ones, as cta_sort leaves it.  is_f32: 32-bit keys are codes of
// floats.  PAIRS: v holds key << 32 | a position that grows with the item's
// place in the unit.  RUNS: the keys are ascending runs of run keys.  MANY:
// units by the thousand, where what a unit costs counts, not how long it takes.
// Ends with __syncthreads().
template <typename K, int T, int E, bool PAIRS = false, bool RUNS = false, bool MANY = false>
__device__ __forceinline__ void cta_bin_sort(K (&v)[E], K *sm, int len, bool is_f32, int run = 0)
{
    using B = BinSort<K, T, E>;
    constexpr int NWARP = B::NWARP, NB = B::NB;
    __shared__ typename std::conditional<PAIRS, uint32_t, K>::type s_lo[NWARP], s_hi[NWARP];
    __shared__ uint32_t s_a[NWARP], s_b[NWARP];
    const B s(sm, len);
    const int lane = s.lane, warp = s.warp;
    // smallest and largest real key; counters to zero
    using V = typename std::conditional<PAIRS, uint32_t, K>::type;
    auto value = [](K x) {
        if constexpr (PAIRS) return (uint32_t)(x >> 32);
        else return x;
    };
    V lo = KeyMax<V>::v, hi = 0;
    if (s.full) {
#pragma unroll
        for (int k = 0; k < E; ++k) {
            lo = kmin<V>(lo, value(v[k]));
            hi = kmax<V>(hi, value(v[k]));
        }
    } else if (s.act) {
#pragma unroll
        for (int k = 0; k < E; ++k)
            if (s.real(k)) {
                lo = kmin<V>(lo, value(v[k]));
                hi = kmax<V>(hi, value(v[k]));
            }
    }
    // (64-bit words by halves)
    auto warp_lo = [&](V x) {
        if constexpr (sizeof(V) == 4) {
            return __reduce_min_sync(0xFFFFFFFFu, x);
        } else {
            const uint32_t h = (uint32_t)(x >> 32), m = __reduce_min_sync(0xFFFFFFFFu, h);
            const uint32_t l = __reduce_min_sync(0xFFFFFFFFu, h == m ? (uint32_t)x : 0xFFFFFFFFu);
            return ((V)m << 32) | l;
        }
    };
    auto warp_hi = [&](V x) {
        if constexpr (sizeof(V) == 4) {
            return __reduce_max_sync(0xFFFFFFFFu, x);
        } else {
            const uint32_t h = (uint32_t)(x >> 32), m = __reduce_max_sync(0xFFFFFFFFu, h);
            const uint32_t l = __reduce_max_sync(0xFFFFFFFFu, h == m ? (uint32_t)x : 0u);
            return ((V)m << 32) | l;
        }
    };
    lo = warp_lo(lo);
    hi = warp_hi(hi);
    if (lane == 0) {
        s_lo[warp] = lo;
        s_hi[warp] = hi;
    }
    uint4 *cnt = s.counters();
    for (int i = s.tid; i < NB / 8; i += T) cnt[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    lo = warp_lo(s_lo[lane % NWARP]);
    hi = warp_hi(s_hi[lane % NWARP]);
    if (hi <= lo) {  // no real key, or all of them equal (pairs: in order)
#pragma unroll
        for (int k = 0; k < E; ++k)
            sm[pidx<K>(wb_pos<E>(warp, lane, k))] = s.real(k) ? v[k] : KeyMax<K>::v;
        __syncthreads();
        return;
    }
    // Keys that crowd into few bins take another sort at once, by the sample.
    // (ANY: small units of 32-bit keys take it for repeated keys too: 6000
    // keys, 1024 values, 14.5 us by comparisons, 21 by bins cut once more; as
    // many 8192-key units 593 us by comparisons, 524 by bins)
    constexpr bool ANY = !PAIRS && sizeof(K) == 4 && B::CAP <= (MANY ? 2048 : 8192);
    const K sx = s.sample(v);
    auto crowding = [&](const auto &map) {
        return s.template crowding<ANY>(map.bin(sx), value(sx));
    };
    auto spill = [&]() {  // the keys to their warp-blocked positions
#pragma unroll
        for (int k = 0; k < E; ++k) sm[pidx<K>(wb_pos<E>(warp, lane, k))] = v[k];
        __syncthreads();
    };
    uint32_t G = 0;
    bool repeated = true;
    // steps 1-3: true when step 4 is still to do
    auto distribute = [&](const auto &map, auto fill) -> bool {
        if (s.full) s.template count<true>(v, map);
        else if (s.act) s.template count<false>(v, map);
        __syncthreads();
        G = s.scan(cnt, cnt, s_a, s_b);
        if constexpr (decltype(fill)::value) {
            if (G > kBinPhases) {
                spill();
                if (!bin_skewed<K, T, E, PAIRS>(sm, len, map, repeated))
                    bin_other<K, T, E, false>(sm, len, 0);
                return false;
            }
        }
        if (s.full) s.template scatter<true>(v, map);
        else if (s.act) s.template scatter<false>(v, map);
        s.pad();
        __syncthreads();
        return decltype(fill)::value;
    };
    // crowded bins that one more cut parts (a quarter of the limit: a few that
    // stay crowded are already too many; the smallest samples are noisier)
    auto parts = [&](const auto &map) -> bool {
        if constexpr (ANY) {
            return false;
        } else {
            repeated =
                s.crowding_cut(map.bin(sx), map.fine(sx), value(sx)) > (T <= 256 ? 0.35f : 0.25f);
            return !repeated;
        }
    };
    auto by_bins = [&](const auto &map, const auto &other) -> bool {
        if (crowding(map) <= 1.0f) return distribute(map, std::true_type{});
        const bool log = !ANY && !(RUNS && run) && !is_f32;
        const float l = log ? crowding(other) : 2.0f;
        if (l > 1.0f && parts(map)) return distribute(map, std::true_type{});
        // (the other map's bins can be cut once more, too)
        if (l <= (T <= 128 ? 1.0f : 1.35f)) {
            spill();
            bin_again<K, T, E, PAIRS>(sm, len, other);
        } else if constexpr (E <= 16 && T <= 512 && (ANY || T <= 256)) {
            cta_sort<K, T, E>(v, sm, len);  // (small: a call would cost a tenth of the sort)
        } else {
            spill();
            bin_other<K, T, E, RUNS>(sm, len, run);
        }
        return false;
    };
    bool more;
    if constexpr (PAIRS) {
        more = by_bins(BinMapPairs<NB>(lo, hi), BinMapLogPairs<NB>(lo, hi));
    } else {
        if (hi - lo < (K)NB) {
            distribute(BinMapExact<K, NB>(lo, hi, lane), std::false_type{});
            return;
        }
        if constexpr (sizeof(K) == 4) {
            // floats: equal steps of the value, or of the code (about its
            // logarithm) where those crowd
            const BinMapF32<NB> fmap(lo, hi);
            bool by_value = is_f32 && fmap.ok;
            if (by_value && crowding(fmap) > 1.0f)
                by_value = crowding(BinMap<uint32_t, NB>(lo, hi)) > 1.0f && parts(fmap);
            if (by_value) more = distribute(fmap, std::true_type{});
            else more = by_bins(BinMap<uint32_t, NB>(lo, hi), BinMapLog<uint32_t, NB>(lo, hi));
        } else {
            more = by_bins(BinMap<K, NB>(lo, hi), BinMapLog<K, NB>(lo, hi));
        }
    }
    if (!more) return;
    s.order_bins(v, G);
}

}  // namespace bsort
