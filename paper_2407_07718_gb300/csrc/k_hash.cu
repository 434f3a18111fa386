// k_hash.cu -- stage S4 + S5 by hashing on chip: the supermer records of a
// bucket are split further by the minimizer's hash into fine partitions, and
// one CTA counts the k-mers of a few partitions at a time in a shared-memory
// table, straight from the records.
//
// A k-mer value never lands in two partitions (all its occurrences share the
// canonical minimizer and so its hash), so partitions are the paper's tasks
// (Sec. 3.4) cut fine enough that the distinct k-mers of one fit an SM.
// The k-mers themselves are never written to memory: a record of 16 (k <= 32)
// or 32 bytes stands for all k-mers of its supermer.
//
//   k_split       -- records of a bucket -> its fine partitions (one CTA per
//                    bucket: count, scan, scatter; no global atomics).
//   k_hash_count  -- per batch of whole partitions: equal records are merged
//                    first (reads of the same locus repeat whole supermers, and
//                    the record of the other strand is the reverse complement),
//                    then the k-mers of each distinct record are added to the
//                    table with the record's multiplicity.  When the table is
//                    full it is emptied: statistics, filter, kept pairs.
//                    Tier 1 is the same kernel with a table of one CTA per SM,
//                    for the partitions that overfill tier 0's; what overfills
//                    that is listed for the sorting path (k_local.cu).
//   k_list_gather -- records of listed partitions -> one array for that path.
//
// What it replaces and measured (one GB300): writing every key to its (group,
// top digit) sub-segment and sorting the sub-segments on chip (k_local.cu)
// took 39 ms on 1.5 G windows of 30x long reads (k = 31) and 45 ms on 1.27 G
// of 20x short reads (k = 55); the split takes 2.1 and 1.3 ms, the counting
// 10.2 and 26.8 ms.
#include "hsk_device.cuh"

namespace hsk {

// ---------------------------------------------------------------------------
// fine partitions
// ---------------------------------------------------------------------------
constexpr int SPLIT_NT = 512;

// Bucket b (first_bucket <= b < last_bucket) holds records
// [bucket_off[b], bucket_off[b+1]) with their sub-partition in rec_sub; they
// go to partitions b * nsub + (sub & (nsub - 1)), in order of partition, at
// out (record bucket_off[first_bucket] first).  part_off receives each
// partition's first record, relative to out.
template <int RW>
__global__ void __launch_bounds__(SPLIT_NT) k_split(const u64* __restrict__ rec, const uint8_t* __restrict__ rec_sub,
                                                    const u64* __restrict__ bucket_off, uint32_t first_bucket,
                                                    uint32_t last_bucket, uint32_t nsub, u64* __restrict__ out,
                                                    u64* __restrict__ part_off) {
    __shared__ uint32_t s_cnt[256];
    __shared__ uint32_t s_scr[SPLIT_NT / 32 + 1];
    const int tid = threadIdx.x;
    const u64 rec0 = bucket_off[first_bucket];
    for (uint32_t b = first_bucket + blockIdx.x; b < last_bucket; b += gridDim.x) {
        const u64 r0 = bucket_off[b];
        const uint32_t n = (uint32_t)(bucket_off[b + 1] - r0);
        const uint8_t* sub = rec_sub + r0;
        if (tid < 256) s_cnt[tid] = 0;
        __syncthreads();
        for (uint32_t i = tid; i < n; i += SPLIT_NT) atomicAdd(&s_cnt[sub[i] & (nsub - 1)], 1u);
        __syncthreads();
        const uint32_t c = tid < 256 ? s_cnt[tid] : 0u;
        uint32_t total;
        const uint32_t e = block_excl_sum<SPLIT_NT, uint32_t>(c, s_scr, total);
        if (tid < 256) s_cnt[tid] = e;
        if (tid < (int)nsub) part_off[(u64)(b - first_bucket) * nsub + tid] = r0 - rec0 + e;
        if (b + 1 == last_bucket && tid == 0) part_off[(u64)(last_bucket - first_bucket) * nsub] = r0 - rec0 + n;
        __syncthreads();
        constexpr int UR = RW == 2 ? 4 : 2;  // records a thread holds at a time
        const ulonglong2* src = reinterpret_cast<const ulonglong2*>(rec + r0 * RW);
        ulonglong2* dst = reinterpret_cast<ulonglong2*>(out + (r0 - rec0) * RW);
        for (uint32_t i0 = tid; i0 < n; i0 += SPLIT_NT * UR) {
            ulonglong2 v[UR][RW / 2];
            uint32_t d[UR];
#pragma unroll
            for (int j = 0; j < UR; ++j) {
                const uint32_t i = i0 + j * SPLIT_NT;
                if (i < n) {
                    d[j] = sub[i] & (nsub - 1);
#pragma unroll
                    for (int q = 0; q < RW / 2; ++q) v[j][q] = src[(size_t)i * (RW / 2) + q];
                }
            }
#pragma unroll
            for (int j = 0; j < UR; ++j) {
                if (i0 + j * SPLIT_NT < n) {
                    const uint32_t at = atomicAdd(&s_cnt[d[j]], 1u);
#pragma unroll
                    for (int q = 0; q < RW / 2; ++q) dst[(size_t)at * (RW / 2) + q] = v[j][q];
                }
            }
        }
        __syncthreads();
    }
}

void launch_split(const uint64_t* records, const uint8_t* rec_sub, const uint64_t* bucket_off, uint32_t first_bucket,
                  uint32_t last_bucket, uint32_t nsub, int rec_words, uint64_t* out, uint64_t* part_off, int num_sms,
                  cudaStream_t st) {
    if (last_bucket <= first_bucket) return;
    count_launch();
    const uint32_t nb = last_bucket - first_bucket;
    const unsigned g = nb < (uint32_t)num_sms * 4 ? nb : (unsigned)num_sms * 4;
    if (rec_words == 2)
        k_split<2><<<g, SPLIT_NT, 0, st>>>((const u64*)records, rec_sub, (const u64*)bucket_off, first_bucket,
                                           last_bucket, nsub, (u64*)out, (u64*)part_off);
    else
        k_split<4><<<g, SPLIT_NT, 0, st>>>((const u64*)records, rec_sub, (const u64*)bucket_off, first_bucket,
                                           last_bucket, nsub, (u64*)out, (u64*)part_off);
}

// ---------------------------------------------------------------------------
// count the k-mers of partitions in a shared-memory table
// ---------------------------------------------------------------------------
// SLOTS table slots (a multiple of NT), RB records per batch, DS slots of the
// record table (a power of two, at least 2 * RB).
template <bool WIDE, int TIER>
struct HashCfg;
template <>
struct HashCfg<false, 0> {
    static constexpr int NT = 512, CTAS = 2, SLOTS = 6656, RB = 1024, DS = 2048;
};
template <>
struct HashCfg<false, 1> {
    static constexpr int NT = 1024, CTAS = 1, SLOTS = 15360, RB = 1024, DS = 2048;
};
template <>
struct HashCfg<true, 0> {
    static constexpr int NT = 512, CTAS = 2, SLOTS = 4096, RB = 512, DS = 1024;
};
template <>
struct HashCfg<true, 1> {
    static constexpr int NT = 512, CTAS = 1, SLOTS = 9216, RB = 512, DS = 1024;
};
constexpr int HC_HS = 128;      // count-histogram bins kept in shared memory
constexpr int HC_SEG = 8;       // k-mers of a record one lane adds at a time
constexpr int HC_CHUNK = 32;    // most partitions claimed at a time
constexpr int HC_PROBES = 512;  // a longer probe sequence means that the table is full
constexpr u64 HC_EMPTY = ~0ULL; // never a stored key word (see insert)
constexpr uint32_t HC_NONE = 0xFFFFFFFFu;

template <bool WIDE, int TIER>
constexpr uint32_t hash_cap() { return HashCfg<WIDE, TIER>::SLOTS / 32 * 27; }  // distinct k-mers held at most

uint32_t hash_count_cap(int key_words) { return key_words == 1 ? hash_cap<false, 0>() : hash_cap<true, 0>(); }

template <bool WIDE, int TIER>
constexpr size_t hash_smem() {
    using C = HashCfg<WIDE, TIER>;
    return (size_t)C::SLOTS * ((WIDE ? 16 : 8) + 4) + (size_t)C::RB * (WIDE ? 32 : 16) + (size_t)C::DS * 4 +
           (size_t)C::RB * 4;
}

// Bases of a record (left aligned, nb of them, the rest 0) reversed and
// complemented, left aligned again.
template <bool WIDE>
__device__ __forceinline__ void record_revcomp(const u64 (&W)[4], uint32_t nb, u64 (&R)[4]) {
    if constexpr (!WIDE) {
        const u64 x0 = reverse_pairs(~W[1]), x1 = reverse_pairs(~W[0]);  // right aligned
        const uint32_t s = 128 - 2 * nb;
        if (s >= 64) {
            R[0] = x1 << (s - 64);  // nb <= 32 here; s = 128 (no bases) does not occur
            R[1] = 0;
        } else {
            R[0] = s ? (x0 << s) | (x1 >> (64 - s)) : x0;
            R[1] = x1 << s;
        }
        R[2] = R[3] = 0;
    } else {
        u64 x[5];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = reverse_pairs(~W[3 - i]);
        x[4] = 0;
        uint32_t s = 256 - 2 * nb;  // < 256
        if (s >= 128) {
            x[0] = x[2];
            x[1] = x[3];
            x[2] = x[3] = 0;
            s -= 128;
        }
        if (s >= 64) {
            x[0] = x[1];
            x[1] = x[2];
            x[2] = x[3];
            x[3] = 0;
            s -= 64;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) R[i] = funnel64(x[i], x[i + 1], s);
    }
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
};

template <bool WIDE, int TIER>
__global__ void __launch_bounds__(HashCfg<WIDE, TIER>::NT, HashCfg<WIDE, TIER>::CTAS)
    k_hash_count(const __grid_constant__ HashArgs P) {
    using Cfg = HashCfg<WIDE, TIER>;
    using K = typename std::conditional<WIDE, key128, u64>::type;
    constexpr int NT = Cfg::NT, NW = NT / 32, SLOTS = Cfg::SLOTS, RB = Cfg::RB, DS = Cfg::DS;
    constexpr int RW = WIDE ? 4 : 2;
    constexpr int RPT = (RB + NT - 1) / NT;  // records a thread stages per batch
    constexpr uint32_t CAP = hash_cap<WIDE, TIER>();
    static_assert(SLOTS % NT == 0 && DS >= 2 * RB && RB <= 1024, "table sizes");
    extern __shared__ __align__(16) unsigned char smem_hc[];
    u64* tk = reinterpret_cast<u64*>(smem_hc);                       // [SLOTS] keys (WIDE: their high words)
    u64* tk2 = tk + SLOTS;                                           // WIDE: [SLOTS] low words
    u64* s_rec = tk + (size_t)SLOTS * (WIDE ? 2 : 1);                // [RB * RW]
    uint32_t* tc = reinterpret_cast<uint32_t*>(s_rec + (size_t)RB * RW);  // [SLOTS] counts
    uint32_t* s_ds = tc + SLOTS;                                     // [DS] record table: index | copies << 16
    uint32_t* s_ord = s_ds + DS;                                     // [RB] distinct records, longest first
    __shared__ uint32_t s_bin[128], s_base[128];                     // distinct records by k-mers; first place of each
    __shared__ uint32_t s_hist[HC_HS], s_dig[256], s_wk[NW];
    __shared__ u64 s_off[HC_CHUNK + 1], s_obase;
    __shared__ uint32_t s_claim, s_U, s_D, s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t hs = P.hist_len < (uint32_t)HC_HS ? P.hist_len : (uint32_t)HC_HS;
    const int k = P.k;

    for (int i = tid; i < SLOTS; i += NT) {
        tk[i] = HC_EMPTY;
        if (WIDE) tk2[i] = HC_EMPTY;
        tc[i] = 0;
    }
    for (int i = tid; i < DS; i += NT) s_ds[i] = HC_NONE;
    for (int i = tid; i < HC_HS; i += NT) s_hist[i] = 0;
    for (int i = tid; i < 256; i += NT) s_dig[i] = 0;
    if (tid < 128) s_bin[tid] = 0;
    if (tid == 0) s_U = s_D = s_fail = 0;
    u64 my_distinct = 0;
    uint32_t my_max = 0, my_ones = 0;

    // Empties the table: every slot is one distinct k-mer with its count.
    auto flush = [&]() {
        uint32_t kept = 0;
        for (int i = tid; i < SLOTS; i += NT) {
            const uint32_t cnt = tc[i];
            if (!cnt) continue;
            ++my_distinct;
            if (cnt == 1) {
                ++my_ones;
            } else {
                const uint32_t b = cnt < P.hist_len - 1 ? cnt : P.hist_len - 1;
                if (b < hs) atomicAdd(&s_hist[b], 1u);
                else atomicAdd(reinterpret_cast<unsigned long long*>(P.hist + b), 1ULL);
            }
            my_max = cnt > my_max ? cnt : my_max;
            kept += (cnt >= P.lo && cnt <= P.hi) ? 1u : 0u;
        }
        kept = __reduce_add_sync(0xffffffffu, kept);
        if (lane == 0) s_wk[warp] = kept;
        __syncthreads();
        if (warp == 0) {
            const uint32_t v = lane < NW ? s_wk[lane] : 0u;
            const uint32_t inc = warp_incl_sum<uint32_t>(v);
            if (lane < NW) s_wk[lane] = inc - v;
            const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
            if (lane == 0) {
                u64 at = total ? atomicAdd(P.out_n, (unsigned long long)total) : 0ULL;
                if (at + total > P.out_cap) {
                    raise_error(P.err, HSK_DERR_BOUNDS);
                    at = HC_EMPTY;
                }
                s_obase = at;
                s_D = 0;
            }
        }
        __syncthreads();
        const bool ok = s_obase != HC_EMPTY;
        u64 at = s_obase + s_wk[warp];
        for (int i = tid; i < SLOTS; i += NT) {
            const uint32_t cnt = tc[i];
            const bool keep = ok && cnt && cnt >= P.lo && cnt <= P.hi;
            const uint32_t km = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                K key;
                if constexpr (WIDE) {
                    const u64 h = tk[i], l = tk2[i];
                    key.hi = h >> 2;
                    key.lo = (h << 62) | l;
                } else {
                    key = tk[i];
                }
                atomicAdd(&s_dig[key_digit(key, P.dshift, 0xFF)], 1u);
                const u64 o = at + (uint32_t)__popc(km & ((1u << lane) - 1u));
                reinterpret_cast<K*>(P.out_keys)[o] = key;
                P.out_counts[o] = cnt;
            }
            at += (uint32_t)__popc(km);
            tk[i] = HC_EMPTY;
            if (WIDE) tk2[i] = HC_EMPTY;
            tc[i] = 0;
        }
        __syncthreads();
    };
    // Empties the table without counting anything (a partition that overfilled it).
    auto discard = [&]() {
        for (int i = tid; i < SLOTS; i += NT) {
            tk[i] = HC_EMPTY;
            if (WIDE) tk2[i] = HC_EMPTY;
            tc[i] = 0;
        }
        if (tid == 0) s_D = s_fail = 0;
        __syncthreads();
    };

    // Records [r0, r0 + nr) into shared memory, each in the smaller of its two
    // orientations, equal ones merged.  Returns the k-mers of the distinct
    // ones (s_U); s_ord lists them, longest first, with their copies.
    auto stage = [&](u64 r0, uint32_t nr) -> uint32_t {
        uint32_t rn[RPT], rr[RPT], rh[RPT];
        uint32_t u = 0;
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
            const uint32_t i = (uint32_t)j * NT + tid;
            rn[j] = 0;
            if (i >= nr) continue;
            u64 W[4] = {0, 0, 0, 0}, R[4];
            const ulonglong2* q = reinterpret_cast<const ulonglong2*>(P.rec + (r0 + i) * RW);
            const ulonglong2 a = q[0];
            W[0] = a.x;
            W[1] = a.y;
            if (WIDE) {
                const ulonglong2 b = q[1];
                W[2] = b.x;
                W[3] = b.y;
            }
            const uint32_t n = (uint32_t)(W[RW - 1] & 0x7F);
            W[RW - 1] &= ~0xFFULL;
            record_revcomp<WIDE>(W, n + k - 1, R);
            bool less = R[0] < W[0];
            if (!WIDE) {
                less = less || (R[0] == W[0] && R[1] < W[1]);
            } else if (R[0] == W[0]) {
                less = R[1] < W[1] || (R[1] == W[1] && (R[2] < W[2] || (R[2] == W[2] && R[3] < W[3])));
            }
            if (less) {
#pragma unroll
                for (int t = 0; t < RW; ++t) W[t] = R[t];
            }
            W[RW - 1] |= n;
            ulonglong2* d = reinterpret_cast<ulonglong2*>(s_rec + (size_t)i * RW);
            d[0] = make_ulonglong2(W[0], W[1]);
            if (WIDE) d[1] = make_ulonglong2(W[2], W[3]);
            __threadfence_block();
            uint32_t x = (uint32_t)W[0] * 0x9E3779B1u + (uint32_t)(W[0] >> 32) * 0x85EBCA77u +
                         (uint32_t)W[1] * 0xC2B2AE3Du + (uint32_t)(W[1] >> 32) * 0x27D4EB2Fu;
            if (WIDE)
                x += (uint32_t)W[2] * 0x165667B1u + (uint32_t)(W[2] >> 32) * 0xD3A2646Du +
                     (uint32_t)W[3] * 0xFD7046C5u + (uint32_t)(W[3] >> 32) * 0xB55A4F09u;
            uint32_t h = (x ^ (x >> 15)) & (DS - 1);
            for (;;) {  // at most RB of the DS slots are taken: this ends
                uint32_t prev = *(volatile uint32_t*)&s_ds[h];
                if (prev == HC_NONE) prev = atomicCAS(&s_ds[h], HC_NONE, i | (1u << 16));
                if (prev == HC_NONE) {
                    rn[j] = n;
                    rh[j] = h;
                    u += n;
                    break;
                }
                const volatile u64* o = s_rec + (size_t)(prev & 0xFFFFu) * RW;
                bool eq = o[0] == W[0] && o[1] == W[1];
                if (WIDE) eq = eq && o[2] == W[2] && o[3] == W[3];
                if (eq) {
                    atomicAdd(&s_ds[h], 1u << 16);
                    break;
                }
                h = (h + 1) & (DS - 1);
            }
            if (rn[j]) rr[j] = atomicAdd(&s_bin[n], 1u);
        }
        u = __reduce_add_sync(0xffffffffu, u);
        if (lane == 0 && u) atomicAdd(&s_U, u);
        __syncthreads();
        if (warp == 0) {  // first place of each length, longest first
            uint32_t c[4], sum = 0;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                c[t] = s_bin[127 - 4 * lane - t];
                sum += c[t];
            }
            uint32_t e = warp_incl_sum<uint32_t>(sum) - sum;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                s_base[127 - 4 * lane - t] = e;
                e += c[t];
            }
        }
        const uint32_t U = s_U;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < RPT; ++j)
            if (rn[j]) s_ord[s_base[rn[j]] + rr[j]] = ((uint32_t)j * NT + tid) | (s_ds[rh[j]] & 0xFFFF0000u);
        if (tid < 128) s_bin[tid] = 0;
        if (tid == 0) s_U = 0;
        __syncthreads();
        for (int i = tid; i < DS; i += NT) s_ds[i] = HC_NONE;
        return U;
    };

    // The k-mers of the staged distinct records into the table.  A warp takes
    // 32 records' k-mers [8 s, 8 s + 8); the order by length keeps its lanes
    // equally busy.  s_base[8 s] is the number of records of more than 8 s
    // k-mers.
    auto insert_all = [&]() {
        uint32_t fresh = 0;
        bool fail = false;
        auto insert = [&](const K& key, uint32_t w) {
            u64 a;
            [[maybe_unused]] u64 b = 0;
            uint32_t x;
            if constexpr (WIDE) {
                // 2 k - 62 and 62 bits: the all-ones word is no low word, and no
                // high word of a canonical code of k <= 63 bases (at k = 63 it
                // would start with 32 T, and so end with 32 A)
                a = (key.hi << 2) | (key.lo >> 62);
                b = key.lo & (~0ULL >> 2);
                x = (uint32_t)b * 0x9E3779B1u + (uint32_t)(b >> 32) * 0x85EBCA77u + (uint32_t)a * 0xC2B2AE3Du +
                    (uint32_t)(a >> 32) * 0x27D4EB2Fu;
            } else {
                a = key;  // never all ones: the reverse complement of all T is smaller
                x = (uint32_t)a * 0x9E3779B1u + (uint32_t)(a >> 32) * 0x85EBCA77u;
            }
            uint32_t h = __umulhi(x, (uint32_t)SLOTS);
            for (int probe = 0; probe < HC_PROBES; ++probe) {
                u64 prev = *(volatile u64*)&tk[h];
                if (prev == HC_EMPTY) {
                    prev = atomicCAS(reinterpret_cast<unsigned long long*>(&tk[h]), HC_EMPTY, a);
                    if (!WIDE && prev == HC_EMPTY) ++fresh;
                }
                bool hit = prev == HC_EMPTY || prev == a;
                if constexpr (WIDE) {
                    // a slot whose high word is set gets its low word from one of
                    // the keys with that high word; the others go on
                    if (hit) {
                        u64 p2 = *(volatile u64*)&tk2[h];
                        if (p2 == HC_EMPTY) {
                            p2 = atomicCAS(reinterpret_cast<unsigned long long*>(&tk2[h]), HC_EMPTY, b);
                            if (p2 == HC_EMPTY) ++fresh;
                        }
                        hit = p2 == HC_EMPTY || p2 == b;
                    }
                }
                if (hit) {
                    atomicAdd(&tc[h], w);
                    return;
                }
                if (++h == (uint32_t)SLOTS) h = 0;
            }
            fail = true;
        };
        uint32_t t = warp;
        for (int s = 0; HC_SEG * s < P.rec_n; ++s) {
            const uint32_t ge = s_base[HC_SEG * s], tiles = (ge + 31) / 32;
            for (; t < tiles; t += NW) {
                if (*(volatile uint32_t*)&s_fail) break;
                const uint32_t q = t * 32 + lane;
                if (q < ge) {
                    const uint32_t e = s_ord[q], i = e & 0xFFFFu, w = e >> 16;
                    u64 W[4] = {0, 0, 0, 0};
                    const ulonglong2* d = reinterpret_cast<const ulonglong2*>(s_rec + (size_t)i * RW);
                    const ulonglong2 a = d[0];
                    W[0] = a.x;
                    W[1] = a.y;
                    if (WIDE) {
                        const ulonglong2 b = d[1];
                        W[2] = b.x;
                        W[3] = b.y;
                    }
                    const uint32_t n = (uint32_t)(W[RW - 1] & 0x7F), j0 = HC_SEG * s;
                    uint32_t sh = 2 * j0;  // drop the first j0 bases
                    while (sh >= 64) {
                        W[0] = W[1];
                        W[1] = W[2];
                        W[2] = W[3];
                        W[3] = 0;
                        sh -= 64;
                    }
                    if (sh) {
#pragma unroll
                        for (int y = 0; y < RW; ++y) W[y] = funnel64(W[y], y < 3 ? W[y + 1] : 0ULL, sh);
                    }
                    const uint32_t nk = n - j0 < (uint32_t)HC_SEG ? n - j0 : (uint32_t)HC_SEG;
                    record_kmers<WIDE>(W, nk, k, [&](uint32_t, const K& key) { insert(key, w); });
                }
            }
            t -= tiles;  // t >= tiles unless the loop stopped on a failure
        }
        fresh = __reduce_add_sync(0xffffffffu, fresh);
        if (lane == 0 && fresh) atomicAdd(&s_D, fresh);
        if (fail) s_fail = 1;
        __syncthreads();
    };

    uint32_t target = RB, D = 0;
    __syncthreads();
    for (;;) {
        if (tid == 0) s_claim = atomicAdd(P.claim, 1u);
        __syncthreads();
        const u64 c0 = (u64)s_claim * P.chunk;
        if (c0 >= P.n_part) break;
        const uint32_t np = P.n_part - c0 < P.chunk ? (uint32_t)(P.n_part - c0) : P.chunk;
        u64 first = c0;
        if (P.only) first = P.only[c0];  // listed partitions are claimed one at a time
        if (tid <= (int)np) s_off[tid] = P.part_off[first + tid];
        __syncthreads();
        for (uint32_t p = 0; p < np;) {
            const u64 r0 = s_off[p];
            uint32_t q = p + 1;
            while (q < np && s_off[q + 1] - r0 <= (u64)target) ++q;
            const u64 nr = s_off[q] - r0;
            if (nr == 0) {
                p = q;
                continue;
            }
            bool over = false;  // more k-mers than the table surely holds: it may overfill
            uint32_t U = 0;
            if (nr <= (u64)RB) {
                U = stage(r0, (uint32_t)nr);
                if (D + U > CAP && D > 0) {
                    flush();
                    D = 0;
                }
                if (U > CAP) {
                    if (q > p + 1) {  // take fewer partitions
                        target = target / 2 > 32 ? target / 2 : 32;
                        __syncthreads();
                        continue;
                    }
                    over = true;
                }
                insert_all();
            } else {  // one partition of more records than fit a batch
                over = true;
                if (D > 0) {
                    flush();
                    D = 0;
                }
                for (u64 r = r0; r < r0 + nr; r += RB) {
                    const u64 left = r0 + nr - r;
                    stage(r, (uint32_t)(left < (u64)RB ? left : (u64)RB));
                    insert_all();
                    if (s_fail) break;
                }
            }
            D = s_D;
            if (over && s_fail) {
                __syncthreads();
                discard();
                D = 0;
                if (tid == 0) {
                    P.ov_list[atomicAdd(reinterpret_cast<unsigned int*>(P.ov_stats), 1u)] = (uint32_t)(first + p);
                    atomicAdd(P.ov_stats + 1, (unsigned long long)nr);
                }
            } else if (s_fail) {  // cannot happen: D + U <= CAP < SLOTS
                if (tid == 0) raise_error(P.err, HSK_DERR_BOUNDS);
                __syncthreads();
                discard();
                D = 0;
            } else if (U < CAP / 3 && target < (uint32_t)RB) {
                target = target * 2 < (uint32_t)RB ? target * 2 : (uint32_t)RB;
            }
            p = q;
        }
        __syncthreads();
    }
    if (D > 0) flush();
    if (my_ones) atomicAdd(&s_hist[1], my_ones);
    __syncthreads();
    for (uint32_t i = tid; i < hs; i += NT)
        if (s_hist[i]) atomicAdd(reinterpret_cast<unsigned long long*>(P.hist + i), (unsigned long long)s_hist[i]);
    for (int i = tid; i < 256; i += NT)
        if (s_dig[i]) atomicAdd(P.dig_hist + i, (unsigned long long)s_dig[i]);
    const u64 d = warp_incl_sum<u64>(my_distinct);
    const uint32_t mx = __reduce_max_sync(0xffffffffu, my_max);
    if (lane == 31 && d) atomicAdd(P.n_distinct, (unsigned long long)d);
    if (lane == 0 && mx) atomicMax(P.max_count, mx);
}

void launch_hash_count(const uint64_t* records, const uint64_t* part_off, const uint32_t* only, uint32_t n_part,
                       int tier, int k, int nmax, uint32_t lo, uint32_t hi, void* out_keys, uint32_t* out_counts,
                       uint64_t out_cap, uint64_t* out_n, uint32_t* ov_list, uint64_t* ov_stats, uint64_t* hist,
                       uint32_t hist_len, uint32_t* max_count, uint64_t* n_distinct, uint64_t* dig_hist,
                       uint32_t* claim, int* err, int num_sms, cudaStream_t st) {
    if (n_part == 0) return;
    count_launch();
    HashArgs P;
    P.rec = (const u64*)records;
    P.part_off = (const u64*)part_off;
    P.only = only;
    P.n_part = n_part;
    P.k = k;
    P.dshift = 2 * k > 8 ? 2 * k - 8 : 0;
    P.rec_n = nmax;
    P.lo = lo;
    P.hi = hi;
    P.out_keys = out_keys;
    P.out_counts = out_counts;
    P.out_cap = out_cap;
    P.out_n = (unsigned long long*)out_n;
    P.ov_list = ov_list;
    P.ov_stats = (unsigned long long*)ov_stats;
    P.hist = (u64*)hist;
    P.hist_len = hist_len;
    P.max_count = max_count;
    P.n_distinct = (unsigned long long*)n_distinct;
    P.dig_hist = (unsigned long long*)dig_hist;
    P.claim = claim;
    P.err = err;
    auto go = [&](auto kern, int nt, int ctas, size_t dyn) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        const uint64_t slots = (uint64_t)num_sms * ctas;
        // enough claims that the CTAs end together, few enough that a claim spans several batches
        uint64_t ch = only ? 1 : n_part / (slots * 8);
        P.chunk = (uint32_t)(ch < 1 ? 1 : ch > HC_CHUNK ? HC_CHUNK : ch);
        const uint64_t want = (n_part + P.chunk - 1) / P.chunk;
        kern<<<(unsigned)(want < slots ? want : slots), nt, dyn, st>>>(P);
    };
#define HC_GO(W, T) go(k_hash_count<W, T>, HashCfg<W, T>::NT, HashCfg<W, T>::CTAS, hash_smem<W, T>())
    if (k <= 32) {
        if (tier) HC_GO(false, 1);
        else HC_GO(false, 0);
    } else {
        if (tier) HC_GO(true, 1);
        else HC_GO(true, 0);
    }
#undef HC_GO
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
