// k_hash.cu -- stage S4 + S5 by hashing on chip: the supermer records come
// scattered into fine partitions (the minimizer's bucket and more bits of its
// hash), and one CTA counts the k-mers of a few partitions at a time in shared
// memory, straight from the records.
//
// A k-mer value never lands in two partitions (all its occurrences share the
// canonical minimizer and so its hash), so partitions are the paper's tasks
// (Sec. 3.4) cut fine enough that the distinct k-mers of one fit an SM.
// The k-mers themselves are never written to memory: a record of 16 (k <= 32)
// or 32 bytes stands for all k-mers of its supermer.
//
//   k_hash_count  -- per batch of whole partitions: equal records are merged
//                    first (reads of the same locus repeat whole supermers;
//                    the records come in one orientation for both strands),
//                    then the k-mers of each distinct record are hashed with
//                    the record's multiplicity, equal ones merged, and the
//                    counts go to the statistics, the filter and the output.
//                    Tier 1 is the same kernel with one CTA per SM and a
//                    larger batch, for partitions that overfill tier 0's.
//   k_pair_merge, k_pair_emit
//                 -- partitions of very many records (reads crowded around one
//                    minimizer), and those that overfill tier 1's table, are cut
//                    into slices that any CTA counts (tier 2 of k_hash_count);
//                    the slices' (k-mer, count) pairs are merged in one table in
//                    global memory.
//   k_list_gather -- records of the partitions whose slices leave too many pairs
//                    -> one array for the sorting path (k_local.cu).
//
// What it replaces and measured (one GB300): writing every key to its (group,
// top digit) sub-segment and sorting the sub-segments on chip (k_local.cu)
// took 39 ms on 1.5 G windows of 30x long reads (k = 31) and 45 ms on 1.27 G
// of 20x short reads (k = 55); this takes 4.6 and 11.5 ms.
#include "hsk_device.cuh"

namespace hsk {

// ---------------------------------------------------------------------------
// count the k-mers of partitions in a shared-memory table
// ---------------------------------------------------------------------------
// A batch holds RB records and ENT k-mers of distinct records at most; 2^LS
// hash slots (of k-mers, and before them of records).
//
// Equal k-mers find each other without a probe sequence: every k-mer of the
// batch has an entry of its own (key, count) and writes its entry's number to
// the slot of its hash.  After a barrier the number in the slot is the
// winner: a k-mer that is not the winner but equal to it adds its count to
// the winner's; one that differs goes to the next round, with another hash.
// All copies of a k-mer take the same slots, so they either merge or go on
// together.  Nothing waits or loops in the first round, which settles most
// k-mers.  What bounds the kernel is instructions and the barriers between
// its phases (about half the issue slots used); an open-addressing table with
// compare-and-swap took three times the instructions, as the lanes of a warp
// wait for its longest probe sequence: 10.2 and 26.8 ms on the two workloads
// above (four tags read at once 10.2 and 27.7), against 4.9 and 13.0.  Visiting
// only the kept entries when the pairs are written (one in nine of the short
// reads') took that to 4.7 and 11.9, the last rounds by one warp to 4.6 and 11.5.
//
// Sizes, by trial.  64-bit keys, on the long reads and on 8x short reads of a
// 20 Mbp genome: 384 threads x 3 CTAs and 3072 entries 5.1 and 0.74 ms, 512 x
// 2 and 4096 5.8 and 0.92, 256 x 4 and 2304 5.5 and 0.77.  128-bit keys, on
// the short reads: 512 x 2 and 3840 entries 12.9 ms, 3584 13.3, 1024 x 1 and
// 7680 14.1.  With the kept entries listed (emit): 3840 12.1 ms, 4032 (what two
// CTAs can hold) 11.9; 64-bit keys 3072 4.72, 3200 4.76.
//
// Tier 1 (and 2), the whole count stage where partitions are overfull.  64-bit keys,
// on 5 Mbp of long reads with repeats and on 30 kb sequenced 20,000 times: 1024
// threads and 8192 entries 0.64 and 1.13 ms, 512 threads 0.65 and 1.18, 512 x 2 CTAs
// and 4864 entries 0.59 and 1.34.  128-bit keys: 512 threads 2.30 and 6.13, 768 2.28
// and 6.09, 1024 2.36 and 6.49.
template <bool WIDE, int TIER>
struct HashCfg;
template <>
struct HashCfg<false, 0> {
    static constexpr int NT = 384, CTAS = 3, ENT = 3072, LS = 13, RB = 768;
};
template <>
struct HashCfg<false, 1> {
    static constexpr int NT = 1024, CTAS = 1, ENT = 8192, LS = 14, RB = 4096;
};
template <>
struct HashCfg<true, 0> {
    static constexpr int NT = 512, CTAS = 2, ENT = 4032, LS = 13, RB = 384;
};
template <>
struct HashCfg<true, 1> {
    static constexpr int NT = 512, CTAS = 1, ENT = 6144, LS = 14, RB = 1536;
};
template <bool WIDE>
struct HashCfg<WIDE, 2> : HashCfg<WIDE, 1> {};
constexpr int HC_HS = 128;      // count-histogram bins kept in shared memory
constexpr int HC_SEG = 16;      // k-mers of a record one lane takes at a time (at most 16)
constexpr int HC_CHUNK = 32;    // most partitions claimed at a time

uint32_t hash_count_cap(int key_words) { return key_words == 1 ? HashCfg<false, 0>::ENT : HashCfg<true, 0>::ENT; }

uint32_t hash_slice_records(int key_words) { return key_words == 1 ? HashCfg<false, 1>::RB : HashCfg<true, 1>::RB; }

template <bool WIDE, int TIER>
constexpr size_t hash_smem() {
    using C = HashCfg<WIDE, TIER>;
    return (size_t)C::ENT * ((WIDE ? 16 : 8) + 4) + (size_t)C::RB * ((WIDE ? 32 : 16) + 4 + 2) + ((size_t)2 << C::LS);
}

// Segment s (HC_SEG k-mers) of a record of 32-bit words w; s is the same in the
// whole warp.
template <bool WIDE>
__device__ __forceinline__ void segment_start(KmerRoll<WIDE>& S, uint32_t (&w)[WIDE ? 8 : 4], int s, int k) {
    constexpr int NW = WIDE ? 8 : 4;
    const int b0 = HC_SEG * s;  // first base
    for (int q = b0 >> 4; q > 0; --q) {
#pragma unroll
        for (int i = 0; i < NW; ++i) w[i] = i + 1 < NW ? w[i + 1] : 0u;
    }
    if (b0 & 15) {
#pragma unroll
        for (int i = 0; i < NW; ++i) w[i] = __funnelshift_l(i + 1 < NW ? w[i + 1] : 0u, w[i], 2 * (b0 & 15));
    }
    S.start(w, k);
}

// Slot (of 2^LS) of a key in round `round`.
template <int LS>
__device__ __forceinline__ uint32_t key_slot(u64 key, uint32_t round) {
    const uint32_t x = (uint32_t)key * 0x9E3779B1u + (uint32_t)(key >> 32) * 0x85EBCA77u;
    return ((x ^ (x >> 15)) * (0x2C1B3C6Du + 2 * round)) >> (32 - LS);
}
template <int LS>
__device__ __forceinline__ uint32_t key_slot(const key128& key, uint32_t round) {
    const uint32_t x = (uint32_t)key.lo * 0x9E3779B1u + (uint32_t)(key.lo >> 32) * 0x85EBCA77u +
                       (uint32_t)key.hi * 0xC2B2AE3Du + (uint32_t)(key.hi >> 32) * 0x27D4EB2Fu;
    return ((x ^ (x >> 15)) * (0x2C1B3C6Du + 2 * round)) >> (32 - LS);
}

struct HashArgs {
    const u64* rec;          // records, partition after partition
    const u64* part_off;     // n_part + 1 (all partitions)
    const uint32_t* only;    // listed partitions (nullptr: 0 .. n_part - 1)
    uint32_t n_part, chunk;  // partitions to count; claimed `chunk` at a time
    int k, dshift, rec_n;    // dshift: shift of a key's top digit
    uint32_t lo, hi;
    void* out_keys;
    uint32_t* out_counts;
    // Sets (packed passes): bucket b belongs to set bucket_set[b] (nullptr: one
    // set); partition p to bucket p >> sub_bits.  Set s's kept pairs go to
    // places out_base[s] .. out_base[s + 1] (one set: 0 .. out_cap), out_n[s] of
    // them, and its statistics to hist + s * hist_len, max_count[s],
    // n_distinct[s] and dig_hist + s * 256.
    const uint32_t* bucket_set;
    int sub_bits;
    const u64* out_base;
    u64 out_cap;
    unsigned long long* out_n;  // kept pairs
    uint32_t* ov_list;
    unsigned long long* ov_stats;  // {partitions listed, their records}
    u64* hist;
    uint32_t hist_len;
    uint32_t* max_count;
    unsigned long long* n_distinct;
    unsigned long long* dig_hist;  // kept pairs per top digit
    uint32_t* claim;
    int* err;
    // Partitions for the slices {first record, records, partition}, while there is
    // room; heavy_n = {listed (or more), records of those in the list}: of tier 0
    // those of more than heavy_min records, of tier 1 all that it cannot take
    u64* heavy;
    u64 heavy_min;
    uint32_t heavy_cap;
    unsigned long long* heavy_n;
    // Tier 2: n_part slices {first record, records, partition}; their pairs (keys
    // left aligned) with their sets (nullptr: one set), pair_n of them or more
    // than pair_cap
    const u64* slice;
    void* pair_keys;
    uint32_t* pair_counts;
    uint32_t* pair_set;
    u64 pair_cap;
    unsigned long long* pair_n;
};

template <bool WIDE, int TIER>
__global__ void __launch_bounds__(HashCfg<WIDE, TIER>::NT, HashCfg<WIDE, TIER>::CTAS)
    k_hash_count(const __grid_constant__ HashArgs P) {
    using Cfg = HashCfg<WIDE, TIER>;
    using K = typename std::conditional<WIDE, key128, u64>::type;
    constexpr int NT = Cfg::NT, NW = NT / 32, ENT = Cfg::ENT, LS = Cfg::LS, RB = Cfg::RB;
    constexpr int RW = WIDE ? 4 : 2;
    constexpr int RPT = (RB + NT - 1) / NT;  // records a thread takes per batch
    static_assert(ENT <= 65536 && RB <= 65536 && (ENT + 3) / 4 <= RB * RW, "16-bit numbers; the lists fit the records' room");
    extern __shared__ __align__(16) unsigned char smem_hc[];
    K* ek = reinterpret_cast<K*>(smem_hc);                           // [ENT] keys, left aligned
    u64* s_rec = reinterpret_cast<u64*>(ek + ENT);                   // [RB * RW] records
    uint16_t* s_list = reinterpret_cast<uint16_t*>(s_rec);           // [ENT] then: entries left for the next round
    uint32_t* ec = reinterpret_cast<uint32_t*>(s_rec + (size_t)RB * RW);  // [ENT] counts
    uint32_t* s_w = ec + ENT;                                        // [RB] copies of a record
    uint16_t* s_slot = reinterpret_cast<uint16_t*>(s_w + RB);        // [2^LS]
    uint16_t* s_ord = s_slot + (1 << LS);                            // [RB] distinct records, longest first
    // distinct records by their number of k-mers; records of more than t k-mers
    // (the first place of t in the order); entry of the first record's k-mer t
    __shared__ uint32_t s_bin[128], s_base[128], s_ent[128];
    __shared__ uint32_t s_hist[HC_HS], s_dig[256], s_wk[NW];
    __shared__ u64 s_off[HC_CHUNK + 1], s_obase;
    __shared__ uint32_t s_claim, s_U, s_nl[2], s_kept;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t hs = P.hist_len < (uint32_t)HC_HS ? P.hist_len : (uint32_t)HC_HS;
    const int k = P.k;
    const u64 mask = ~0ULL << (WIDE ? 128 - 2 * k : 64 - 2 * k);  // a left-aligned key's (low) word

    for (int i = tid; i < HC_HS; i += NT) s_hist[i] = 0;
    for (int i = tid; i < 256; i += NT) s_dig[i] = 0;
    if (tid < 128) s_bin[tid] = 0;
    if (tid < 2) s_nl[tid] = 0;
    uint32_t my_max = 0, my_ones = 0, my_more = 0;  // largest count; k-mers seen once, more often
    if (tid == 0) s_kept = 0;
    uint32_t set = 0;  // the set whose statistics are held here
    u64 out0 = 0, out1 = P.out_cap;
    if (P.bucket_set) {
        out0 = P.out_base[0];
        out1 = P.out_base[1];
    }
    u64* hist = P.hist;

    // Records [r0, r0 + nr) into shared memory, equal ones merged (most of
    // them: a record that meets another one in its slot stays distinct).
    // Returns the k-mers of the distinct ones; when they fit, s_ord lists
    // those records, longest first.
    auto stage = [&](u64 r0, uint32_t nr) -> uint32_t {
        uint32_t rn[RPT], rr[RPT];  // k-mers | slot << 16 of this thread's records; place among equal lengths
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
            const uint32_t i = (uint32_t)j * NT + tid;
            rn[j] = 0;
            if (i >= nr) continue;
            const uint4* src = reinterpret_cast<const uint4*>(P.rec + (r0 + i) * RW);
            uint4* dst = reinterpret_cast<uint4*>(s_rec + (size_t)i * RW);
            const uint4 a = src[0];
            dst[0] = a;
            uint32_t x = a.x * 0x9E3779B1u + a.y * 0x85EBCA77u + a.z * 0xC2B2AE3Du + a.w * 0x27D4EB2Fu;
            uint32_t n = a.z & 0x7Fu;
            if (WIDE) {
                const uint4 b = src[1];
                dst[1] = b;
                x += b.x * 0x165667B1u + b.y * 0xD3A2646Du + b.z * 0xFD7046C5u + b.w * 0xB55A4F09u;
                n = b.z & 0x7Fu;
            }
            const uint32_t h = ((x ^ (x >> 15)) * 0x2C1B3C6Du) >> (32 - LS);
            *(volatile uint16_t*)&s_slot[h] = (uint16_t)i;
            s_w[i] = 1;
            rn[j] = n | (h << 16);
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
            const uint32_t i = (uint32_t)j * NT + tid, n = rn[j] & 0xFFFFu;
            if (i >= nr) continue;
            const uint32_t win = s_slot[rn[j] >> 16];
            if (win != i) {
                const uint4* a = reinterpret_cast<const uint4*>(s_rec + (size_t)i * RW);
                const uint4* b = reinterpret_cast<const uint4*>(s_rec + (size_t)win * RW);
                const uint4 u = a[0], v = b[0];
                bool eq = u.x == v.x && u.y == v.y && u.z == v.z && u.w == v.w;
                if (WIDE && eq) {
                    const uint4 u1 = a[1], v1 = b[1];
                    eq = u1.x == v1.x && u1.y == v1.y && u1.z == v1.z && u1.w == v1.w;
                }
                if (eq) {
                    atomicAdd(&s_w[win], 1u);
                    rn[j] = 0;
                    continue;
                }
            }
            rr[j] = atomicAdd(&s_bin[n], 1u);
        }
        __syncthreads();
        if (warp == 0) {
            // s_base[t] = records of more than t k-mers, s_ent[t] = its sum over the t before
            uint32_t c[4], sum = 0;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                c[t] = s_bin[127 - 4 * lane - t];
                sum += c[t];
            }
            uint32_t e = warp_incl_sum<uint32_t>(sum) - sum;
            sum = 0;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                s_base[127 - 4 * lane - t] = e;
                sum += e;
                e += c[t];
                c[t] = e - c[t];
            }
            const uint32_t inc = warp_incl_sum<uint32_t>(sum);
            const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
            uint32_t g = total - inc;
#pragma unroll
            for (int t = 3; t >= 0; --t) {
                s_ent[127 - 4 * lane - t] = g;
                g += c[t];
            }
            if (lane == 0) s_U = total;
        }
        __syncthreads();
        const uint32_t U = s_U;
        if (tid < 128) s_bin[tid] = 0;
        if (U <= (uint32_t)ENT) {
#pragma unroll
            for (int j = 0; j < RPT; ++j)
                if (rn[j] & 0xFFFFu) s_ord[s_base[rn[j] & 0xFFFFu] + rr[j]] = (uint16_t)((uint32_t)j * NT + tid);
        }
        __syncthreads();
        return U;
    };

    // The k-mers of the staged distinct records: key, count and slot of each.
    // A warp takes 32 records' k-mers [HC_SEG s, HC_SEG s + HC_SEG); the order
    // by length keeps its lanes equally busy, and k-mer t of the q-th record
    // is entry D + s_ent[t] + q, so the lanes write side by side.
    auto expand = [&](uint32_t D) {
        uint32_t t = warp;
        for (int s = 0; HC_SEG * s < P.rec_n; ++s) {
            const uint32_t ge = s_base[HC_SEG * s], tiles = (ge + 31) / 32;
            for (; t < tiles; t += NW) {
                const uint32_t q = t * 32 + lane;
                if (q < ge) {
                    const uint32_t i = s_ord[q], w = s_w[i];
                    uint32_t W[2 * RW];
                    const uint4* d = reinterpret_cast<const uint4*>(s_rec + (size_t)i * RW);
#pragma unroll
                    for (int y = 0; y < RW / 2; ++y) {  // words of 64 bits, low half first
                        const uint4 v = d[y];
                        W[4 * y] = v.y;
                        W[4 * y + 1] = v.x;
                        W[4 * y + 2] = v.w;
                        W[4 * y + 3] = v.z;
                    }
                    const int nk = min((int)(W[2 * RW - 1] & 0x7Fu) - HC_SEG * s, HC_SEG);
                    KmerRoll<WIDE> S;
                    segment_start<WIDE>(S, W, s, k);
                    for (int j = 0; j < nk; ++j) {
                        const K key = S.left(mask);
                        S.step();
                        const uint32_t own = D + s_ent[HC_SEG * s + j] + q;
                        ek[own] = key;
                        ec[own] = w;
                        *(volatile uint16_t*)&s_slot[key_slot<LS>(key, 0)] = (uint16_t)own;
                    }
                }
            }
            t -= tiles;
        }
    };

    // Entry i after its slot was written: merged into the winner, or listed
    // for the next round.
    auto settle = [&](uint32_t i, uint32_t round, uint32_t* nl) {
        const K key = ek[i];
        const uint32_t win = s_slot[key_slot<LS>(key, round)];
        if (win != i) {
            if (key_eq(ek[win], key)) {
                atomicAdd(&ec[win], ec[i]);
                ec[i] = 0;
            } else {
                s_list[atomicAdd(nl, 1u)] = (uint16_t)i;
            }
        }
    };
    // Merges equal k-mers of U entries.
    auto merge = [&](uint32_t U) {
        for (uint32_t i = tid; i < U; i += NT) settle(i, 0, &s_nl[0]);
        __syncthreads();
        for (uint32_t round = 1;; ++round) {  // at least one key a slot is settled every round
            const uint32_t nl = s_nl[(round - 1) & 1];
            if (nl == 0) break;
            // the last few: one warp, without the CTA's barriers (long reads 4.73 ->
            // 4.60 ms, short reads 11.9 -> 11.5; 32 4.63, 128 4.59, 256 4.73)
            if (nl <= 64) {
                if (warp == 0) {
                    uint32_t e[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const uint32_t q = 32 * j + lane;
                        e[j] = q < nl ? s_list[q] : 0xFFFFFFFFu;
                    }
                    for (uint32_t r = round;; ++r) {
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            if (e[j] != 0xFFFFFFFFu) *(volatile uint16_t*)&s_slot[key_slot<LS>(ek[e[j]], r)] = (uint16_t)e[j];
                        __syncwarp();
                        bool left = false;
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            if (e[j] == 0xFFFFFFFFu) continue;
                            const K key = ek[e[j]];
                            const uint32_t win = *(volatile uint16_t*)&s_slot[key_slot<LS>(key, r)];
                            if (win == e[j]) {
                                e[j] = 0xFFFFFFFFu;
                            } else if (key_eq(ek[win], key)) {
                                atomicAdd(&ec[win], ec[e[j]]);
                                ec[e[j]] = 0;
                                e[j] = 0xFFFFFFFFu;
                            } else {
                                left = true;
                            }
                        }
                        if (!__any_sync(0xffffffffu, left)) break;
                        __syncwarp();
                    }
                }
                __syncthreads();
                break;
            }
            // this thread's entries, in registers: the list is written again
            constexpr int LPT = (ENT + NT - 1) / NT;
            uint32_t e[LPT];
#pragma unroll
            for (int j = 0; j < LPT; ++j) {
                const uint32_t q = (uint32_t)j * NT + tid;
                e[j] = q < nl ? s_list[q] : 0xFFFFFFFFu;
                if (q < nl) *(volatile uint16_t*)&s_slot[key_slot<LS>(ek[e[j]], round)] = (uint16_t)e[j];
            }
            if (tid == 0) s_nl[round & 1] = 0;
            __syncthreads();
#pragma unroll
            for (int j = 0; j < LPT; ++j)
                if (e[j] != 0xFFFFFFFFu) settle(e[j], round, &s_nl[round & 1]);
            __syncthreads();
        }
        if (tid < 2) s_nl[tid] = 0;  // read next after later barriers
    };

    // Statistics, filter and kept pairs of the U merged entries (count 0:
    // merged into another).  The kept ones are listed, so that only they are
    // visited again.
    auto emit = [&](uint32_t U) {
        for (uint32_t i0 = 0; i0 < U; i0 += NT) {
            const uint32_t i = i0 + tid;
            const uint32_t cnt = i < U ? ec[i] : 0u;
            if (cnt > 1) {
                const uint32_t b = cnt < P.hist_len - 1 ? cnt : P.hist_len - 1;
                if (b < hs) atomicAdd(&s_hist[b], 1u);
                else atomicAdd(reinterpret_cast<unsigned long long*>(hist + b), 1ULL);
                ++my_more;
            }
            my_ones += cnt == 1 ? 1u : 0u;
            my_max = cnt > my_max ? cnt : my_max;
            const bool keep = cnt && cnt >= P.lo && cnt <= P.hi;
            const uint32_t km = __ballot_sync(0xffffffffu, keep);
            if (km) {
                uint32_t at = 0;
                if (lane == 0) at = atomicAdd(&s_kept, (uint32_t)__popc(km));
                at = __shfl_sync(0xffffffffu, at, 0);
                if (keep) s_list[at + (uint32_t)__popc(km & ((1u << lane) - 1u))] = (uint16_t)i;
            }
        }
        __syncthreads();
        const uint32_t kept = s_kept;
        if (kept == 0) return;
        if (tid == 0) {
            u64 at = out0 + atomicAdd(P.out_n + set, (unsigned long long)kept);
            if (at + kept > out1) {
                raise_error(P.err, HSK_DERR_BOUNDS);
                at = ~0ULL;
            }
            s_obase = at;
        }
        __syncthreads();
        const u64 at = s_obase;
        if (tid == 0) s_kept = 0;
        if (at == ~0ULL) return;
        for (uint32_t q = tid; q < kept; q += NT) {
            const uint32_t i = s_list[q];
            const K key = right_aligned(ek[i], k);
            atomicAdd(&s_dig[key_digit(key, P.dshift, 0xFF)], 1u);
            reinterpret_cast<K*>(P.out_keys)[at + q] = key;
            P.out_counts[at + q] = ec[i];
        }
    };

    // The held statistics to their set; leaves them cleared.
    auto flush_stats = [&]() {
        if (my_ones) atomicAdd(&s_hist[1], my_ones);  // hist_len >= 2: count 1 has its own bin
        __syncthreads();
        for (uint32_t i = tid; i < hs; i += NT) {
            if (s_hist[i]) atomicAdd(reinterpret_cast<unsigned long long*>(hist + i), (unsigned long long)s_hist[i]);
            s_hist[i] = 0;
        }
        for (int i = tid; i < 256; i += NT) {
            if (s_dig[i]) atomicAdd(P.dig_hist + (u64)set * 256 + i, (unsigned long long)s_dig[i]);
            s_dig[i] = 0;
        }
        const u64 d = warp_incl_sum<u64>((u64)my_ones + my_more);
        const uint32_t mx = __reduce_max_sync(0xffffffffu, my_max);
        if (lane == 31 && d) atomicAdd(P.n_distinct + set, (unsigned long long)d);
        if (lane == 0 && mx) atomicMax(P.max_count + set, mx);
        my_max = my_ones = my_more = 0;
        __syncthreads();
    };
    // Moves the entries in use to the front; returns their number.
    auto close_up = [&](uint32_t D) -> uint32_t {
        uint32_t at = 0;
        for (uint32_t i0 = 0; i0 < D; i0 += NT) {  // in order: no entry is overwritten before it is read
            const uint32_t i = i0 + tid;
            const uint32_t cnt = i < D ? ec[i] : 0u;
            K key{};
            if (cnt) key = ek[i];
            const uint32_t m = __ballot_sync(0xffffffffu, cnt != 0);
            if (lane == 0) s_wk[warp] = (uint32_t)__popc(m);
            __syncthreads();
            uint32_t pos = at;
            for (int w = 0; w < NW; ++w) {
                if (w < warp) pos += s_wk[w];
                at += s_wk[w];
            }
            if (cnt) {
                pos += (uint32_t)__popc(m & ((1u << lane) - 1u));
                ek[pos] = key;
                ec[pos] = cnt;
            }
            __syncthreads();
        }
        return at;
    };
    // records of a part: what fills half the room at U k-mers in n records
    auto next_part = [&](uint32_t n, uint32_t U, uint32_t room) -> uint32_t {
        const uint32_t t = (uint32_t)((u64)n * room / (2 * (u64)U));
        return t < 16 ? 16 : t >= n ? (n > 32 ? n / 2 : 16) : t;
    };
    // One partition of more than a batch, in parts: the distinct k-mers of the
    // parts so far keep their entries (closed up when room runs out), and every
    // part's are merged with them.  False when even those do not fit.
    auto count_in_parts = [&](u64 r0, u64 nr, uint32_t U) -> bool {
        uint32_t D = 0, take = (uint32_t)(nr < (u64)RB ? nr : (u64)RB);
        if (U != 0xFFFFFFFFu) take = next_part(take, U, ENT);
        for (u64 r = r0; r < r0 + nr;) {
            const uint32_t n = r0 + nr - r < (u64)take ? (uint32_t)(r0 + nr - r) : take;
            U = stage(r, n);
            if (D + U > (uint32_t)ENT) {
                const uint32_t before = D;
                D = close_up(D);
                if (D + U > (uint32_t)ENT) {  // a smaller part, unless the entries are nearly all distinct k-mers
                    if (D > (uint32_t)ENT / 4 * 3 || (before == D && n <= 16)) return false;
                    take = next_part(n, U, (uint32_t)ENT - D);
                    continue;
                }
            }
            expand(D);
            for (uint32_t i = tid; i < D; i += NT) *(volatile uint16_t*)&s_slot[key_slot<LS>(ek[i], 0)] = (uint16_t)i;
            __syncthreads();
            merge(D + U);
            __syncthreads();
            D += U;
            r += n;
        }
        emit(D);
        __syncthreads();
        return true;
    };
    // records of the next batch: as many as fill 15/16 of the entries at the
    // last batch's k-mers per record
    auto next_target = [&](uint32_t nr, uint32_t U) -> uint32_t {
        const uint32_t t = nr * (uint32_t)(ENT / 16 * 15) / (U ? U : 1u);  // nr <= 4096, ENT <= 8192: no overflow
        return t > (uint32_t)RB ? (uint32_t)RB : t;
    };
    if constexpr (TIER == 2) {
        // the D entries as pairs
        auto put_pairs = [&](uint32_t D) {
            D = close_up(D);
            if (tid == 0) s_obase = atomicAdd(P.pair_n, (unsigned long long)D);
            __syncthreads();
            const u64 at = s_obase;
            if (at + D <= P.pair_cap)
                for (uint32_t i = tid; i < D; i += NT) {
                    reinterpret_cast<K*>(P.pair_keys)[at + i] = ek[i];
                    P.pair_counts[at + i] = ec[i];
                    if (P.pair_set) P.pair_set[at + i] = set;
                }
            __syncthreads();
        };
        for (;;) {
            __syncthreads();
            if (tid == 0) s_claim = atomicAdd(P.claim, 1u);
            __syncthreads();
            if (s_claim >= P.n_part) break;
            const u64* sl = P.slice + 3 * (u64)s_claim;
            u64 r = sl[0];
            const u64 end = r + sl[1];
            if (P.bucket_set) set = P.bucket_set[sl[2] >> P.sub_bits];
            uint32_t D = 0, take = RB;
            while (r < end) {
                if (tid == 0) s_kept = *(volatile unsigned long long*)P.pair_n > P.pair_cap;
                __syncthreads();
                if (s_kept) break;  // too many pairs already: all are dropped
                const uint32_t n = end - r < (u64)take ? (uint32_t)(end - r) : take;
                const uint32_t U = stage(r, n);
                if (D + U > (uint32_t)ENT) D = close_up(D);
                if (D + U > (uint32_t)ENT && D > (uint32_t)ENT / 2) {
                    put_pairs(D);
                    D = 0;
                }
                if (D + U > (uint32_t)ENT) {  // more than 16 records: those have fewer k-mers than half the entries
                    take = next_part(n, U, (uint32_t)ENT - D);
                    continue;
                }
                expand(D);
                for (uint32_t i = tid; i < D; i += NT) *(volatile uint16_t*)&s_slot[key_slot<LS>(ek[i], 0)] = (uint16_t)i;
                __syncthreads();
                merge(D + U);
                __syncthreads();
                D += U;
                r += n;
                // about three eighths of the entries a part
                const uint32_t t = n * (uint32_t)(ENT / 8 * 3) / (U ? U : 1u);
                take = t < 16 ? 16 : t > (uint32_t)RB ? (uint32_t)RB : t;
            }
            put_pairs(D);
        }
        return;
    }
    uint32_t target = RB;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_claim = atomicAdd(P.claim, 1u);
        __syncthreads();
        const u64 c0 = (u64)s_claim * P.chunk;
        if (c0 >= P.n_part) break;
        const uint32_t np = P.n_part - c0 < P.chunk ? (uint32_t)(P.n_part - c0) : P.chunk;
        u64 first = c0;
        if (P.only) first = P.only[c0];  // listed partitions are claimed one at a time
        if (tid <= (int)np) s_off[tid] = P.part_off[first + tid];
        if (P.bucket_set) {  // a claim lies within one bucket
            const uint32_t now = P.bucket_set[first >> P.sub_bits];
            if (now != set) {
                flush_stats();
                set = now;
                out0 = P.out_base[set];
                out1 = P.out_base[set + 1];
                hist = P.hist + (u64)set * P.hist_len;
            }
        }
        __syncthreads();
        for (uint32_t p = 0; p < np;) {
            // the batch: as many whole partitions as `target` records hold
            const u64 r0 = s_off[p];
            uint32_t q = p + 1;
            while (q < np && s_off[q + 1] - r0 <= (u64)target) ++q;
            const u64 nr = s_off[q] - r0;
            if (nr == 0) {
                p = q;
                continue;
            }
            uint32_t U = nr <= (u64)RB ? stage(r0, (uint32_t)nr) : 0xFFFFFFFFu;
            if (U > (uint32_t)ENT) {
                if (q > p + 1) {  // take fewer partitions
                    target = next_target((uint32_t)nr, U);
                    if (target >= (uint32_t)nr) target = (uint32_t)nr - 1;
                    continue;
                }
                // partition p alone is more than a batch
                if (TIER == 0 || !count_in_parts(r0, nr, U)) {
                    if (tid == 0) {
                        u64 at = P.heavy_cap;
                        if (TIER == 1 || nr > P.heavy_min) at = atomicAdd(P.heavy_n, 1ULL);
                        if (at < (u64)P.heavy_cap) {
                            P.heavy[3 * at] = r0;
                            P.heavy[3 * at + 1] = nr;
                            P.heavy[3 * at + 2] = first + p;
                            atomicAdd(P.heavy_n + 1, (unsigned long long)nr);
                        } else {
                            P.ov_list[atomicAdd(reinterpret_cast<unsigned int*>(P.ov_stats), 1u)] = (uint32_t)(first + p);
                            atomicAdd(P.ov_stats + 1, (unsigned long long)nr);
                        }
                    }
                    __syncthreads();
                }
                ++p;
                continue;
            }
            expand(0);
            __syncthreads();
            merge(U);
            emit(U);
            __syncthreads();
            target = next_target((uint32_t)nr, U);
            p = q;
        }
    }
    flush_stats();
}

template <bool WIDE, int TIER>
static void go_hash_count(HashArgs& P, int num_sms, cudaStream_t st) {
    using C = HashCfg<WIDE, TIER>;
    const size_t dyn = hash_smem<WIDE, TIER>();
    cudaFuncSetAttribute(k_hash_count<WIDE, TIER>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    const uint64_t slots = (uint64_t)num_sms * C::CTAS;
    // enough claims that the CTAs end together, few enough that a claim spans several batches
    uint64_t ch = P.only || TIER == 2 ? 1 : P.n_part / (slots * 8);
    if (ch < 1) ch = 1;
    if (ch > HC_CHUNK) ch = HC_CHUNK;
    if (P.bucket_set) {  // a power of two, at most a bucket's partitions
        uint64_t c2 = 1;
        while (c2 * 2 <= ch && c2 * 2 <= (1ull << P.sub_bits)) c2 *= 2;
        ch = c2;
    }
    P.chunk = (uint32_t)ch;
    const uint64_t want = (P.n_part + P.chunk - 1) / P.chunk;
    k_hash_count<WIDE, TIER><<<(unsigned)(want < slots ? want : slots), C::NT, dyn, st>>>(P);
}

static HashArgs hash_args(const HashJob& J) {
    HashArgs P{};
    P.rec = (const u64*)J.records;
    P.part_off = (const u64*)J.part_off;
    P.k = J.k;
    P.dshift = 2 * J.k > 8 ? 2 * J.k - 8 : 0;
    P.rec_n = J.nmax;
    P.lo = J.lo;
    P.hi = J.hi;
    P.out_keys = J.out_keys;
    P.out_counts = J.out_counts;
    P.bucket_set = J.bucket_set;
    P.sub_bits = J.sub_bits;
    P.out_base = (const u64*)J.out_base;
    P.out_cap = J.out_cap;
    P.out_n = (unsigned long long*)J.out_n;
    P.hist = (u64*)J.hist;
    P.hist_len = J.hist_len;
    P.max_count = J.max_count;
    P.n_distinct = (unsigned long long*)J.n_distinct;
    P.dig_hist = (unsigned long long*)J.dig_hist;
    P.err = J.err;
    return P;
}

void launch_hash_count(const HashJob& J, const uint32_t* only, uint32_t n_part, int tier, uint32_t* ov_list,
                       uint64_t* ov_stats, uint64_t* heavy, uint32_t heavy_cap, uint64_t heavy_min, uint64_t* heavy_n,
                       uint32_t* claim, int num_sms, cudaStream_t st) {
    if (n_part == 0) return;
    count_launch();
    HashArgs P = hash_args(J);
    P.only = only;
    P.n_part = n_part;
    P.ov_list = ov_list;
    P.ov_stats = (unsigned long long*)ov_stats;
    P.heavy = (u64*)heavy;
    P.heavy_min = heavy_min;
    P.heavy_cap = heavy_cap;
    P.heavy_n = (unsigned long long*)heavy_n;
    P.claim = claim;
    if (J.k <= 32) tier ? go_hash_count<false, 1>(P, num_sms, st) : go_hash_count<false, 0>(P, num_sms, st);
    else tier ? go_hash_count<true, 1>(P, num_sms, st) : go_hash_count<true, 0>(P, num_sms, st);
}

void launch_hash_slices(const HashJob& J, const uint64_t* slices, uint32_t n_slices, void* pair_keys,
                        uint32_t* pair_counts, uint32_t* pair_set, uint64_t pair_cap, uint64_t* pair_n,
                        uint32_t* claim, int num_sms, cudaStream_t st) {
    if (n_slices == 0) return;
    count_launch();
    HashArgs P = hash_args(J);
    P.slice = (const u64*)slices;
    P.n_part = n_slices;
    P.pair_keys = pair_keys;
    P.pair_counts = pair_counts;
    P.pair_set = pair_set;
    P.pair_cap = pair_cap;
    P.pair_n = (unsigned long long*)pair_n;
    P.claim = claim;
    if (J.k <= 32) go_hash_count<false, 2>(P, num_sms, st);
    else go_hash_count<true, 2>(P, num_sms, st);
}

// ---------------------------------------------------------------------------
// pairs of the slices -> counts of k-mers
// ---------------------------------------------------------------------------
// Merges equal k-mers (of one set) of n pairs: every pair looks for its k-mer in
// an open-addressing table of pair numbers (+ 1), zeroed, with twice as many slots
// as pairs; the one that enters it keeps the sum, the others end with count 0.
// Bound by the table's random accesses.  With the slices it counts 150 Mbp of
// 150-base reads of one base with 1 % errors in 0.4 and 2.4 ms (k = 31 and 55),
// where one CTA took 30 and 81; one 400-base amplicon (150 Mbp) in 0.6 and 3.1,
// where most of it went on to the sorting path (4.1 and 23 ms in all).
template <typename K>
__global__ void __launch_bounds__(256) k_pair_merge(const K* __restrict__ keys, uint32_t* counts,
                                                    const uint32_t* __restrict__ sets, uint32_t n, uint32_t* table,
                                                    uint32_t mask, int* err) {
    for (uint32_t i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        const K key = keys[i];
        const uint32_t cnt = counts[i], set = sets ? sets[i] : 0u;
        uint32_t h = key_slot<32>(key, 0) ^ set * 0x9E3779B1u;
        h = (h ^ (h >> 16)) & mask;
        for (uint32_t probe = 0;; ++probe) {
            if (probe > mask) {  // never: the table has twice as many slots as pairs
                raise_error(err, HSK_DERR_BOUNDS);
                break;
            }
            const uint32_t v = atomicCAS(&table[h], 0u, i + 1);
            if (v == 0) break;
            if (key_eq(keys[v - 1], key) && (!sets || sets[v - 1] == set)) {
                atomicAdd(&counts[v - 1], cnt);
                counts[i] = 0;
                break;
            }
            h = (h + 1) & mask;
        }
    }
}

// Statistics, filter and kept pairs of n merged pairs (as k_hash_count's emit).
// A CTA takes a run of pairs; pairs of one set lie together in slices, so tiles
// of several sets, which go to memory pair by pair, are few.
template <typename K>
__global__ void __launch_bounds__(256) k_pair_emit(const __grid_constant__ HashArgs P, uint32_t n) {
    __shared__ uint32_t s_hist[HC_HS], s_dig[256], s_n;
    __shared__ u64 s_at;
    const int tid = threadIdx.x, lane = tid & 31;
    const K* keys = reinterpret_cast<const K*>(P.pair_keys);
    const uint32_t hs = P.hist_len < (uint32_t)HC_HS ? P.hist_len : (uint32_t)HC_HS;
    const uint32_t i0 = (uint32_t)((u64)n * blockIdx.x / gridDim.x), i1 = (uint32_t)((u64)n * (blockIdx.x + 1) / gridDim.x);
    if (i0 >= i1) return;
    uint32_t set = P.pair_set ? P.pair_set[i0] : 0u, my_max = 0, my_n = 0;
    for (int i = tid; i < HC_HS; i += 256) s_hist[i] = 0;
    s_dig[tid] = 0;
    if (tid == 0) s_n = 0;
    auto bin_of = [&](uint32_t c) { return c < P.hist_len - 1 ? c : P.hist_len - 1; };
    auto flush = [&]() {
        __syncthreads();
        for (uint32_t i = tid; i < hs; i += 256) {
            if (s_hist[i]) atomicAdd((unsigned long long*)(P.hist + (u64)set * P.hist_len + i), (unsigned long long)s_hist[i]);
            s_hist[i] = 0;
        }
        if (s_dig[tid]) atomicAdd(P.dig_hist + (u64)set * 256 + tid, (unsigned long long)s_dig[tid]);
        s_dig[tid] = 0;
        const uint32_t d = __reduce_add_sync(0xffffffffu, my_n), mx = __reduce_max_sync(0xffffffffu, my_max);
        if (lane == 0 && d) atomicAdd(P.n_distinct + set, (unsigned long long)d);
        if (lane == 0 && mx) atomicMax(P.max_count + set, mx);
        my_n = my_max = 0;
        __syncthreads();
    };
    __syncthreads();
    for (uint32_t b = i0; b < i1; b += 256) {
        const uint32_t i = b + tid;
        const uint32_t cnt = i < i1 ? P.pair_counts[i] : 0u;
        const bool keep = cnt && cnt >= P.lo && cnt <= P.hi;
        const uint32_t mine = cnt && P.pair_set ? P.pair_set[i] : set;
        if (!__syncthreads_and(mine == set)) {
            flush();
            if (cnt) {
                atomicAdd((unsigned long long*)(P.hist + (u64)mine * P.hist_len + bin_of(cnt)), 1ULL);
                atomicAdd(P.n_distinct + mine, 1ULL);
                atomicMax(P.max_count + mine, cnt);
            }
            if (keep) {
                const K key = right_aligned(keys[i], P.k);
                const u64 at = P.out_base[mine] + atomicAdd(P.out_n + mine, 1ULL);
                atomicAdd(P.dig_hist + (u64)mine * 256 + key_digit(key, P.dshift, 0xFF), 1ULL);
                if (at < P.out_base[mine + 1]) {
                    reinterpret_cast<K*>(P.out_keys)[at] = key;
                    P.out_counts[at] = cnt;
                } else {
                    raise_error(P.err, HSK_DERR_BOUNDS);
                }
            }
            set = P.pair_set[i1 - b > 256 ? b + 255 : i1 - 1];
            continue;
        }
        if (cnt) {
            const uint32_t c = bin_of(cnt);
            if (c < hs) atomicAdd(&s_hist[c], 1u);
            else atomicAdd((unsigned long long*)(P.hist + (u64)set * P.hist_len + c), 1ULL);
            ++my_n;
            my_max = cnt > my_max ? cnt : my_max;
        }
        const uint32_t km = __ballot_sync(0xffffffffu, keep);
        uint32_t q = 0;
        if (lane == 0 && km) q = atomicAdd(&s_n, (uint32_t)__popc(km));
        q = __shfl_sync(0xffffffffu, q, 0) + (uint32_t)__popc(km & ((1u << lane) - 1u));
        __syncthreads();
        if (tid == 0) {
            const u64 base = P.bucket_set ? P.out_base[set] : 0, top = P.bucket_set ? P.out_base[set + 1] : P.out_cap;
            u64 at = s_n ? base + atomicAdd(P.out_n + set, (unsigned long long)s_n) : 0;
            if (at + s_n > top) {
                raise_error(P.err, HSK_DERR_BOUNDS);
                at = ~0ULL;
            }
            s_at = at;
            s_n = 0;
        }
        __syncthreads();
        if (keep && s_at != ~0ULL) {
            const K key = right_aligned(keys[i], P.k);
            atomicAdd(&s_dig[key_digit(key, P.dshift, 0xFF)], 1u);
            reinterpret_cast<K*>(P.out_keys)[s_at + q] = key;
            P.out_counts[s_at + q] = cnt;
        }
    }
    flush();
}

void launch_pairs(const HashJob& J, void* pair_keys, uint32_t* pair_counts, uint32_t* pair_set, uint32_t n,
                  uint32_t* table, uint32_t mask, int num_sms, cudaStream_t st) {
    if (n == 0) return;
    count_launch(2);
    HashArgs P = hash_args(J);
    P.pair_keys = pair_keys;
    P.pair_counts = pair_counts;
    P.pair_set = pair_set;
    const uint32_t want = (n + 255) / 256, most = (uint32_t)num_sms * 8, g = want < most ? want : most;
    if (J.k <= 32) {
        k_pair_merge<u64><<<g, 256, 0, st>>>((const u64*)pair_keys, pair_counts, pair_set, n, table, mask, J.err);
        k_pair_emit<u64><<<g, 256, 0, st>>>(P, n);
    } else {
        k_pair_merge<key128><<<g, 256, 0, st>>>((const key128*)pair_keys, pair_counts, pair_set, n, table, mask, J.err);
        k_pair_emit<key128><<<g, 256, 0, st>>>(P, n);
    }
}

// ---------------------------------------------------------------------------
// the sets' kept pairs -> one after the other
// ---------------------------------------------------------------------------
// dst pairs [dst_off[s], dst_off[s + 1]) = src pairs from src_off[s] on.
template <typename K>
__global__ void __launch_bounds__(256) k_close_sets(const K* __restrict__ ks, const uint32_t* __restrict__ cs,
                                                    const u64* __restrict__ src_off, const u64* __restrict__ dst_off,
                                                    uint32_t n_sets, K* __restrict__ kd, uint32_t* __restrict__ cd) {
    const u64 n = dst_off[n_sets];
    for (u64 b = (u64)blockIdx.x * 2048; b < n; b += (u64)gridDim.x * 2048) {
        for (u64 i = b + threadIdx.x; i < b + 2048 && i < n; i += 256) {
            uint32_t lo = 0, hi = n_sets;  // dst_off[lo] <= i < dst_off[hi]
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if (dst_off[mid] <= i) lo = mid;
                else hi = mid;
            }
            const u64 q = src_off[lo] + (i - dst_off[lo]);
            kd[i] = ks[q];
            cd[i] = cs[q];
        }
    }
}

void launch_close_sets(const void* src_keys, const uint32_t* src_counts, const uint64_t* src_off,
                       const uint64_t* dst_off, uint32_t n_sets, uint64_t n, int key_words, void* dst_keys,
                       uint32_t* dst_counts, int num_sms, cudaStream_t st) {
    if (n == 0) return;
    count_launch();
    const uint64_t want = (n + 2047) / 2048;
    const unsigned g = (unsigned)(want < (uint64_t)num_sms * 8 ? want : (uint64_t)num_sms * 8);
    if (key_words == 1)
        k_close_sets<u64><<<g, 256, 0, st>>>((const u64*)src_keys, src_counts, (const u64*)src_off,
                                             (const u64*)dst_off, n_sets, (u64*)dst_keys, dst_counts);
    else
        k_close_sets<key128><<<g, 256, 0, st>>>((const key128*)src_keys, src_counts, (const u64*)src_off,
                                                (const u64*)dst_off, n_sets, (key128*)dst_keys, dst_counts);
}

// ---------------------------------------------------------------------------
// listed partitions -> one array of records
// ---------------------------------------------------------------------------
// CTA j copies the records of partition list[j] to dst + dst_off[j] and sums their k-mers.
template <int RW>
__global__ void __launch_bounds__(256) k_list_gather(const u64* __restrict__ rec, const u64* __restrict__ part_off,
                                                     const uint32_t* __restrict__ list, uint32_t n_list,
                                                     const u64* __restrict__ dst_off, u64* __restrict__ dst,
                                                     unsigned long long* __restrict__ kmers) {
    for (uint32_t j = blockIdx.x; j < n_list; j += gridDim.x) {
        const u64 r0 = part_off[list[j]], n = part_off[list[j] + 1] - r0, o = dst_off[j];
        u64 sum = 0;
        for (u64 i = threadIdx.x; i < n; i += 256) {
#pragma unroll
            for (int q = 0; q < RW; ++q) {
                const u64 w = rec[(r0 + i) * RW + q];
                dst[(o + i) * RW + q] = w;
                if (q == RW - 1) sum += w & 0xFF;
            }
        }
        sum = warp_incl_sum<u64>(sum);
        if ((threadIdx.x & 31) == 31 && sum) atomicAdd(kmers + j, (unsigned long long)sum);
    }
}

void launch_list_gather(const uint64_t* records, const uint64_t* part_off, const uint32_t* list, uint32_t n_list,
                        const uint64_t* dst_off, uint64_t* dst, uint64_t* kmers, int rec_words, int num_sms,
                        cudaStream_t st) {
    if (n_list == 0) return;
    count_launch();
    const unsigned g = n_list < (uint32_t)num_sms * 8 ? n_list : (unsigned)num_sms * 8;
    if (rec_words == 2)
        k_list_gather<2><<<g, 256, 0, st>>>((const u64*)records, (const u64*)part_off, list, n_list,
                                            (const u64*)dst_off, (u64*)dst, (unsigned long long*)kmers);
    else
        k_list_gather<4><<<g, 256, 0, st>>>((const u64*)records, (const u64*)part_off, list, n_list,
                                            (const u64*)dst_off, (u64*)dst, (unsigned long long*)kmers);
}

}  // namespace hsk
