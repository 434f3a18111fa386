// k_supermer.cu -- stages S2 and S3: canonical k-mers, hash-scored minimizers
// and supermers scattered into minimizer-hashed buckets.
//
// Sec. 3.2: every m-mer is scored by a hash (MurmurHash3's 32-bit finalizer
// of the canonical m-mer folded to 32 bits, XOR a seed); a k-mer's minimizer
// is its lowest-scoring m-mer, and the same hash value decides the k-mer's
// target: bucket = score mod B (B a power of two).  Sec. 2.4: consecutive
// k-mers with the same target form a supermer whose overlapping bases are
// stored once.  Sec. 3.4: the buckets are the paper's tasks -- a k-mer value
// never lands in two of them, because canonical m-mers give a k-mer and its
// reverse complement the same minimizer score.
//
// GPU design (replaces the paper's per-read monotone deque): a warp walks a
// tile of 1024 consecutive window starts, lane l the 32 windows that start in
// its 64-bit word of packed bases.  The tile's bases and masks are staged in
// shared memory with 128-bit loads.  A lane computes its 32 m-mer scores from
// two words by constant shifts, then the minima of runs of D scores (D the
// largest power of two <= w) by doubling in registers; a window's minimum is
// that of two overlapping runs.  Supermer cuts (bucket change, invalid window,
// cap of nmax k-mers, tile end) are bit masks of the lane's windows: a
// supermer starts where a bit is set, and ends at the next set bit of the
// cuts, in this lane or a later one.  Every supermer becomes an 8-byte
// descriptor (start base, k-mer count, bucket), appended to a global list with
// one atomic per tile (or two, when S3 takes the buckets in two halves);
// per-bucket record and k-mer counts are kept in shared memory.  A second, light
// kernel scatters records into their buckets from the descriptors.  DUMP mode
// writes per-window keys and scores for the stage test.
//
// The kernel is bound by the integer pipe (ncu: 75 % busy, 67 thread
// instructions per window).  With 32 windows a lane it takes 3.7 ms on 1.5 G
// windows of long reads (k = 31, w = 15) and 4.6 ms on 1.27 G of short reads (k
// = 55, w = 35), with 32 warps a CTA; 8 warps and three CTAs per SM took 4.4 and
// 5.4 ms (64 registers allow 32 warps per SM instead of 24, for some 140 bytes a
// thread spilled, and one table serves them all).  One window a lane and step, with the window minima and the
// cuts found by shuffles and ballots across lanes, took 8.7 warp instructions
// per window and 14.4 and 17.0 ms.  Right shifts done by the multiply pipe (12 %
// busy) made no difference.
#include "hsk_device.cuh"

namespace hsk {

constexpr int SM_TW = 32 * 32;            // windows per warp tile, 32 per lane
constexpr int SM_PW = SM_TW / 32 + 6;     // packed words staged per warp (even)
constexpr int SM_MW = SM_TW / 64 + 4;     // mask words staged per warp (even)
constexpr int SM_ROWS = 33 * 33;          // words of run minima per warp (33 padded rows of 32)
constexpr int SM_VW = SM_TW / 64;         // valid-window words per warp
static_assert(SM_TW == (int)SM_TILE_BASES, "tile size");
static_assert(SM_PW * 32 <= (int)SM_TILE_REACH && SM_MW * 64 <= (int)SM_TILE_REACH,
              "a tile's staged words must lie within its declared reach");

// The bucket table sets the walk's shared memory, so it differs from call to
// call.  Serving slots launch the walk from several host threads at once, and
// the per-kernel opt-in limit is process-wide: every thread sets it to the
// size of the largest table (SM_MAX_BUCKETS buckets), never to its own, so
// one thread cannot lower it under another's launch.
constexpr uint32_t SM_MAX_BUCKETS = 8192;
size_t supermer_smem_bytes(int mode, uint32_t n_buckets, int warps) {
    size_t s = (size_t)warps * ((SM_PW + 2 * SM_MW + SM_VW) * sizeof(u64) + SM_ROWS * sizeof(uint32_t));
    if (mode == SM_DESC) s += (size_t)n_buckets * 2 * sizeof(uint32_t);
    return s;
}

// MurmurHash3's 32-bit finalizer (A. Appleby, public domain).
__device__ __forceinline__ uint32_t fmix32(uint32_t h) {
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}

// Score of the m-mer at local base q of the staged words.  Hash order (the
// paper's choice, Sec. 3.2): MurmurHash3's finalizer of the canonical m-mer.
// Lexical order (the alternative the paper compares against): the canonical
// m-mer's code itself -- its top 32 bits when m > 16, so that the score stays
// 32-bit (m-mers sharing their first 16 bases then tie, which only groups them
// in one bucket).  Either way the score is a function of the canonical m-mer,
// so a k-mer and its reverse complement share their minimizer and bucket.
template <bool LEX>
__device__ __forceinline__ uint32_t mmer_score(const u64* pk, int q, int m, uint32_t seed) {
    u64 f = extract_k64(pk, (u64)q, m);
    u64 r = revcomp64(f, m);
    u64 c = f < r ? f : r;
    if constexpr (LEX) return m > 16 ? (uint32_t)(c >> (2 * m - 32)) : (uint32_t)c;
    else return fmix32((uint32_t)c ^ (uint32_t)(c >> 32) ^ seed);
}

// Bits [2*nb, 64) of word x cleared when the record holds only nb (< 32) more bases.
__device__ __forceinline__ u64 keep_bases(u64 x, int nb) {
    if (nb >= 32) return x;
    if (nb <= 0) return 0;
    return x & (~0ULL << (64 - 2 * nb));
}

// Descriptor of a supermer, from its combined bucket b = bucket | sub << 13.
// Plain: start base (40 bits), k-mers (8), bucket (16).  With fine partitions:
// start base (36), k-mers (7), bucket (13), sub-partition (8).
__device__ __forceinline__ u64 make_desc(u64 pos, uint32_t n, uint32_t b, bool fine) {
    return fine ? pos | ((u64)n << 36) | ((u64)b << 43) : pos | ((u64)n << 40) | ((u64)b << 48);
}

// Window minima of a tile.  Lane l holds the scores of positions 32 l .. 32 l
// + 31 in a[0..31] and in h0, h1 those of positions 1024 + l and 1056 + l (h1
// only read when w > 33).  With D = 2^L <= w < 2 D the minimum of a window is
// that of two overlapping runs of D scores; the run minima come from doubling
// in registers, and the entries past the lane's own 32 from the next lane
// (its first d at level d), exchanged through rows of 33 words (lane l's word
// j at l * 33 + j: no bank conflicts; row 32 holds the positions past the
// tile).  Leaves the run minima in the rows too, and returns the distance of
// the two runs; the window minimum of position j is then
// min(row[j], row[j + off]) (row_at).
__device__ __forceinline__ int run_minima(uint32_t (&a)[32], uint32_t h0, uint32_t h1, int w, uint32_t* rows, int lane) {
    uint32_t* own = rows + lane * 33;
    const uint32_t* nxt = own + 33;
    int D = 1;
#pragma unroll
    for (int d = 1; d <= 16; d *= 2) {
        if (2 * d <= w) {
#pragma unroll
            for (int j = 0; j < d; ++j) own[j] = a[j];
            if (lane < d) rows[32 * 33 + lane] = h0;
            __syncwarp();
            uint32_t n[16];
#pragma unroll
            for (int j = 0; j < d; ++j) n[j] = nxt[j];
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 32; ++j) a[j] = min(a[j], j + d < 32 ? a[j + d < 32 ? j + d : 0] : n[j + d < 32 ? 0 : j + d - 32]);
            const uint32_t o0 = __shfl_sync(0xffffffffu, h0, (lane + d) & 31);
            const uint32_t o1 = __shfl_sync(0xffffffffu, h1, (lane + d) & 31);
            h0 = min(h0, lane + d < 32 ? o0 : o1);
            if (lane + d < 32) h1 = min(h1, o1);
            D = 2 * d;
        }
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) own[j] = a[j];
    rows[32 * 33 + lane] = h0;
    __syncwarp();
    if (w >= 64) {
        uint32_t n[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) n[j] = nxt[j];
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 32; ++j) own[j] = a[j] = min(a[j], n[j]);
        rows[32 * 33 + lane] = min(h0, h1);
        __syncwarp();
        D = 64;
    }
    return w - D;
}
// word of position 32 * lane + j (j < 63) in the rows
__device__ __forceinline__ uint32_t row_at(const uint32_t* rows, int lane, int j) {
    return rows[lane * 33 + j + (j >= 32 ? 1 : 0)];
}

// Scores of the 32 m-mers starting in word W0 of the packed bases (W1 the next
// word).  The forward codes are funnels of W0:W1 by constant shifts; the
// reverse complements are funnels of the reversed and complemented words,
// shifted once so that those shifts are constant too.  Codes stay left
// aligned with the following bases below them: two codes that differ compare
// by their own bits, and equal ones are the same m-mer.  For m > 16 the first
// 16 bases decide: an m-mer and its reverse complement that agree there (base i
// and base m - 1 - i are complements for every i < 16, and m <= 32) are equal,
// and the code's low word comes from the words shifted by the other m - 16 bases.
template <bool SHORT, bool LEX>
__device__ __forceinline__ void mmer_scores32(u64 W0, u64 W1, int m, uint32_t seed, uint32_t (&a)[32]) {
    u64 R0 = reverse_pairs(~W1), R1 = reverse_pairs(~W0);
    auto shift = [](u64& h, u64& l, uint32_t s) {  // s in 0 .. 64
        if (s == 64) {
            h = l;
            l = 0;
        } else if (s) {
            h = (h << s) | (l >> (64 - s));
            l <<= s;
        }
    };
    shift(R0, R1, 2 * (33 - m));
    const uint32_t F[5] = {(uint32_t)(W0 >> 32), (uint32_t)W0, (uint32_t)(W1 >> 32), (uint32_t)W1, 0u};
    const uint32_t C[5] = {(uint32_t)(R0 >> 32), (uint32_t)R0, (uint32_t)(R1 >> 32), (uint32_t)R1, 0u};
    if constexpr (SHORT || LEX) {
        const int sh = SHORT ? 32 - 2 * m : 0;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            const int fi = j / 16, fs = 2 * (j % 16), ci = (31 - j) / 16, cs = 2 * ((31 - j) % 16);
            const uint32_t c = min(__funnelshift_l(F[fi + 1], F[fi], fs), __funnelshift_l(C[ci + 1], C[ci], cs)) >> sh;
            a[j] = LEX ? c : fmix32(c ^ seed);
        }
    } else {
        shift(W0, W1, 2 * (m - 16));
        shift(R0, R1, 2 * (m - 16));
        const uint32_t G[5] = {(uint32_t)(W0 >> 32), (uint32_t)W0, (uint32_t)(W1 >> 32), (uint32_t)W1, 0u};
        const uint32_t E[5] = {(uint32_t)(R0 >> 32), (uint32_t)R0, (uint32_t)(R1 >> 32), (uint32_t)R1, 0u};
        const int sh = 64 - 2 * m;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            const int fi = j / 16, fs = 2 * (j % 16), ci = (31 - j) / 16, cs = 2 * ((31 - j) % 16);
            const uint32_t fh = __funnelshift_l(F[fi + 1], F[fi], fs), ch = __funnelshift_l(C[ci + 1], C[ci], cs);
            const uint32_t fl = __funnelshift_l(G[fi + 1], G[fi], fs), cl = __funnelshift_l(E[ci + 1], E[ci], cs);
            a[j] = fmix32((fh < ch ? fl : cl) ^ (min(fh, ch) >> sh) ^ seed);
        }
    }
}

template <int MODE, bool SHORT, bool LEX, bool FINE, bool TWO_ENDED>
__global__ void __launch_bounds__(SM_CTA_WARPS * 32, 1) k_supermer(const __grid_constant__ SmParams P) {
    extern __shared__ __align__(16) unsigned char smem[];
    u64* s_pk = reinterpret_cast<u64*>(smem);
    const int warps = blockDim.x >> 5;
    u64* s_iv = s_pk + warps * SM_PW;
    u64* s_rs = s_iv + warps * SM_MW;
    u64* s_val = s_rs + warps * SM_MW;
    uint32_t* s_rows = reinterpret_cast<uint32_t*>(s_val + warps * SM_VW);
    uint32_t* s_km = s_rows + warps * SM_ROWS;  // DESC: k-mers per bucket
    uint32_t* s_cnt = s_km + P.n_buckets;       // DESC without fine partitions: records per bucket

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t B = P.n_buckets;
    const int k = P.k, m = P.m, w = P.w, nmax = P.nmax;

    if (MODE == SM_DESC) {
        for (uint32_t b = threadIdx.x; b < (FINE ? B : 2 * B); b += blockDim.x) s_km[b] = 0;
        __syncthreads();
    }

    u64* wpk = s_pk + warp * SM_PW;
    u64* wiv = s_iv + warp * SM_MW;
    u64* wrs = s_rs + warp * SM_MW;
    u64* wval = s_val + warp * SM_VW;
    uint32_t* rows = s_rows + warp * SM_ROWS;
    const u64 n_tiles = P.tile_end ? P.tile_end : (P.n_bases + SM_TW - 1) / SM_TW;

    for (u64 t = P.tile_begin + (u64)blockIdx.x * warps + warp; t < n_tiles; t += (u64)gridDim.x * warps) {
        const u64 p0 = t * SM_TW;
        // buckets of the tile's set (packed sets: the set holding tile t)
        uint32_t bbase = 0, bmask = B - 1u;
        if (P.n_sets) {
            uint32_t lo = 0, hi = P.n_sets;  // set_tile0[lo] <= t < set_tile0[hi]
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if ((u64)P.set_tile0[mid] <= t) lo = mid;
                else hi = mid;
            }
            bbase = P.set_bucket[lo];
            bmask = P.set_bmask[lo];
        }
        // ---- stage packed bases and masks (128-bit loads; p0 is 1024-aligned)
        {
            const u64 pw0 = p0 >> 5, mw0 = p0 >> 6;
            for (int i = lane; i < SM_PW / 2; i += 32) {
                u64 g = pw0 + 2 * i;
                ulonglong2 v = make_ulonglong2(0, 0);
                if (g + 1 < P.n_packed_words) v = *reinterpret_cast<const ulonglong2*>(P.packed + g);
                else if (g < P.n_packed_words) v.x = P.packed[g];
                wpk[2 * i] = v.x;
                wpk[2 * i + 1] = v.y;
            }
            for (int i = lane; i < SM_MW / 2; i += 32) {
                u64 g = mw0 + 2 * i;
                ulonglong2 a = make_ulonglong2(~0ULL, ~0ULL), b = make_ulonglong2(0, 0);
                if (g + 1 < P.n_mask_words) {
                    a = *reinterpret_cast<const ulonglong2*>(P.invalid + g);
                    b = *reinterpret_cast<const ulonglong2*>(P.start + g);
                } else if (g < P.n_mask_words) {
                    a.x = P.invalid[g];
                    b.x = P.start[g];
                }
                wiv[2 * i] = a.x;
                wiv[2 * i + 1] = a.y;
                wrs[2 * i] = b.x;
                wrs[2 * i + 1] = b.y;
            }
            __syncwarp();
            // window starts of the tile whose k bases are all valid and in one
            // read: no invalid base in [p, p+k), no read start in (p, p+k)
            if (lane < SM_TW / 64) {
                const int o = lane;
                u64 bad = window_or64(wiv[o], wiv[o + 1], k);
                if (k > 1) {
                    const u64 a = (wrs[o] << 1) | (wrs[o + 1] >> 63);
                    const u64 b = (wrs[o + 1] << 1) | (wrs[o + 2] >> 63);
                    bad |= window_or64(a, b, k - 1);
                }
                wval[o] = ~bad;
            }
            __syncwarp();
        }
        // valid windows of this lane, window j at bit j
        const u64 v64 = wval[lane >> 1];
        uint32_t V = __brev(lane & 1 ? (uint32_t)v64 : (uint32_t)(v64 >> 32));
        {
            const u64 p = p0 + 32 * lane + k;  // end of window 0
            const u64 left = P.n_bases + 1 > p ? P.n_bases + 1 - p : 0;  // windows that end inside the data
            if (left < 32) V &= (1u << left) - 1u;
        }

        uint32_t a[32];
        mmer_scores32<SHORT, LEX>(wpk[lane], wpk[lane + 1], m, P.seed32, a);
        const uint32_t h0 = mmer_score<LEX>(wpk, SM_TW + lane, m, P.seed32);
        const uint32_t h1 = w > 33 ? mmer_score<LEX>(wpk, SM_TW + 32 + lane, m, P.seed32) : 0xFFFFFFFFu;
        const int off = run_minima(a, h0, h1, w, rows, lane);

        if (MODE == SM_DUMP) {
            for (int j = 0; j < 32; ++j) {
                const u64 p = p0 + 32 * lane + j;
                if (p >= P.n_bases) break;
                const bool valid = (V >> j) & 1u;
                P.dump_valid[p] = valid;
                if (!valid) continue;
                if (k <= 32) {
                    P.dump_key[2 * p] = canonical64(extract_k64(wpk, 32 * lane + j, k), k);
                    P.dump_key[2 * p + 1] = 0;
                } else {
                    const key128 c = canonical128(extract_k128(wpk, 32 * lane + j, k), k);
                    P.dump_key[2 * p] = c.lo;
                    P.dump_key[2 * p + 1] = c.hi;
                }
                P.dump_minhash[p] = min(row_at(rows, lane, j), row_at(rows, lane, j + off));
            }
        } else {
            // id of a window: its bucket and, with fine partitions, the hash bits
            // above it; D has bit j set where window j's id differs from window j - 1's
            const int bb = __popc(bmask);
            const uint32_t idmask = (((bmask + 1u) << P.sub_bits) - 1u);
            uint32_t D = 0, prev = 0;
            [[maybe_unused]] uint32_t late = 0;  // bit j: the lowest bit of window j's id
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const uint32_t id = min(a[j], row_at(rows, lane, j + off)) & idmask;
                if (j > 0) D |= id != prev ? 1u << j : 0u;
                else a[0] = id;
                if (TWO_ENDED) late = __funnelshift_r(late, id, 1);
                prev = id;
            }
            const uint32_t before = __shfl_up_sync(0xffffffffu, prev, 1);
            const uint32_t vb = __shfl_up_sync(0xffffffffu, V, 1);
            D |= a[0] != before ? 1u : 0u;
            const uint32_t Vp = (V << 1) | (lane ? vb >> 31 : 0u);  // window before is valid (and in the tile)
            const uint32_t start = V & (D | ~Vp);
            const uint32_t ev = start | ~V;  // a run that is open here ends
            // the first such place after this lane's windows, in the tile
            const uint32_t has = __ballot_sync(0xffffffffu, ev != 0);
            const uint32_t later = lane < 31 ? has >> (lane + 1) << (lane + 1) : 0u;
            const int nl = later ? __ffs(later) - 1 : lane;
            const int fe = __shfl_sync(0xffffffffu, __ffs(ev) - 1, nl);
            const int open_end = later ? 32 * nl + fe : SM_TW;
            // descriptors: all upward from the array's start, or (TWO_ENDED)
            // those of windows with the lowest id bit set downward from its end;
            // `mine` and its sums hold the numbers of the two in 16 bits each
            uint32_t mine = (uint32_t)__popc(start);
            if (TWO_ENDED) mine += 0xFFFFu * (uint32_t)__popc(start & late);
            const uint32_t incl = warp_incl_sum<uint32_t>(mine);
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
            if (total) {
                u64 at0 = 0, at1 = 0;
                auto reserve = [&](uint32_t sum, uint32_t n) {  // this lane's places, from its exclusive sum
                    const uint32_t n0 = TWO_ENDED ? n & 0xFFFFu : n, n1 = TWO_ENDED ? n >> 16 : 0u;
                    if (lane == 0 && n0) at0 = atomicAdd(P.desc_count, (unsigned long long)n0);
                    if (lane == 0 && n1) at1 = atomicAdd(P.desc_count + 1, (unsigned long long)n1);
                    at0 = __shfl_sync(0xffffffffu, at0, 0) + (TWO_ENDED ? sum & 0xFFFFu : sum);
                    if (TWO_ENDED) at1 = __shfl_sync(0xffffffffu, at1, 0) + (sum >> 16);
                };
                reserve(incl - mine, total);
                uint32_t extra = 0;  // pieces past the first of runs of more than nmax k-mers, counted like `mine`
                // TWO_ENDED: the id's lowest bit is the bucket's highest, so the two
                // kinds are the two halves of the records
                auto bucket_of = [&](uint32_t id) {
                    const uint32_t in = id & bmask;
                    return bbase + (TWO_ENDED ? (in >> 1) | ((in & 1u) << (bb - 1)) : in);
                };
                auto part_of = [&](uint32_t id, uint32_t b) { return (b << P.sub_bits) | (id >> bb); };
                auto put = [&](int pos, int n, uint32_t id, uint32_t b) {
                    const bool down = TWO_ENDED && (id & 1u);
                    const u64 at = down ? P.desc_cap - 1 - at1++ : at0++;  // past the capacity: not written
                    if (at < P.desc_cap)
                        P.desc[at] = make_desc(p0 + pos, (uint32_t)n, b | (id >> bb) << 13, FINE);
                };
                // Records per fine partition: one atomic for all pieces of a run, and the
                // records of the first window's partition added up over the tile.  Reads
                // crowded around one minimizer have nearly all of theirs there, and an
                // atomic per record queues at its address, 1.3 a nanosecond: 150 Mbp of
                // one-base reads took 3.3 ms (now 0.45), with 1 % errors 3.8 (now 0.58).
                // Other reads pay 3 % of the walk for it, and get as much back from kernels
                // of their own for fine partitions.
                [[maybe_unused]] const uint32_t id0 = min(rows[0], row_at(rows, 0, off)) & idmask;
                [[maybe_unused]] const uint32_t hot = part_of(id0, bucket_of(id0));
                [[maybe_unused]] uint32_t hot_n = 0;
                for (uint32_t S = start; S; S &= S - 1) {
                    const int j = __ffs(S) - 1;
                    const uint32_t rest = ev & ~((2u << j) - 1u);
                    const int len = (rest ? 32 * lane + __ffs(rest) - 1 : open_end) - (32 * lane + j);
                    const uint32_t id = min(row_at(rows, lane, j), row_at(rows, lane, j + off)) & idmask;
                    const uint32_t b = bucket_of(id);
                    uint32_t n_rec = 1;
                    if (len > nmax) {
                        const uint32_t more = (uint32_t)((len - 1) / nmax);
                        extra += more << (TWO_ENDED && (id & 1u) ? 16 : 0);
                        n_rec += more;
                    }
                    if (FINE) {
                        const uint32_t part = part_of(id, b);
                        if (part == hot) hot_n += n_rec;
                        else atomicAdd(P.part_rec + part, n_rec);
                    } else {
                        atomicAdd(&s_cnt[b], n_rec);
                    }
                    atomicAdd(&s_km[b], (uint32_t)len);
                    put(32 * lane + j, min(len, nmax), id, b);
                }
                if (FINE) {
                    hot_n = __reduce_add_sync(0xffffffffu, hot_n);
                    if (lane == 0 && hot_n) atomicAdd(P.part_rec + hot, hot_n);
                }
                if (__any_sync(0xffffffffu, extra)) {
                    const uint32_t xi = warp_incl_sum<uint32_t>(extra);
                    at0 = at1 = 0;
                    reserve(xi - extra, __shfl_sync(0xffffffffu, xi, 31));
                    for (uint32_t S = extra ? start : 0u; S; S &= S - 1) {
                        const int j = __ffs(S) - 1;
                        const uint32_t rest = ev & ~((2u << j) - 1u);
                        const int end = rest ? 32 * lane + __ffs(rest) - 1 : open_end;
                        const uint32_t id = min(row_at(rows, lane, j), row_at(rows, lane, j + off)) & idmask;
                        const uint32_t b = bucket_of(id);
                        for (int q = 32 * lane + j + nmax; q < end; q += nmax) put(q, min(end - q, nmax), id, b);
                    }
                }
            }
        }
        __syncwarp();
    }

    if (MODE == SM_DESC) {
        __syncthreads();
        for (uint32_t b = threadIdx.x; b < B; b += blockDim.x) {
            if (!FINE && s_cnt[b]) atomicAdd(P.bucket_rec + b, s_cnt[b]);
            if (s_km[b]) atomicAdd(reinterpret_cast<unsigned long long*>(P.bucket_kmers + b),
                                   (unsigned long long)s_km[b]);
        }
    }
}

using SmKernel = void (*)(SmParams);
template <int MODE, bool FINE, bool TWO_ENDED>
static SmKernel walk_kernel(int m, bool lexical) {
    if (m <= 16)
        return lexical ? (SmKernel)k_supermer<MODE, true, true, FINE, TWO_ENDED>
                       : (SmKernel)k_supermer<MODE, true, false, FINE, TWO_ENDED>;
    return lexical ? (SmKernel)k_supermer<MODE, false, true, FINE, TWO_ENDED>
                   : (SmKernel)k_supermer<MODE, false, false, FINE, TWO_ENDED>;
}
static SmKernel walk_kernel(int mode, int m, bool lexical, bool fine, bool two_ended) {
    SmKernel fn = mode != SM_DESC ? walk_kernel<SM_DUMP, false, false>(m, lexical)
                  : two_ended     ? walk_kernel<SM_DESC, true, true>(m, lexical)
                  : fine          ? walk_kernel<SM_DESC, true, false>(m, lexical)
                                  : walk_kernel<SM_DESC, false, false>(m, lexical);
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)supermer_smem_bytes(mode, SM_MAX_BUCKETS, SM_CTA_WARPS));
    return fn;
}

void launch_supermer(int mode, const SmParams& p, cudaStream_t st) {
    if (p.n_bases == 0) return;
    count_launch();
    walk_kernel(mode, p.m, p.lexical, p.part_rec != nullptr, p.two_ended)<<<p.grid, p.warps * 32, supermer_smem_bytes(mode, p.n_buckets, p.warps), st>>>(p);
}

// As many warps a CTA as leave every SM one (at most SM_CTA_WARPS, at least 4):
// the CTA's table of bucket counters, and adding it up at the end, is shared by
// its warps.  One CTA of 16, 20, 24 and 32 warps per SM took 4.2, 3.9, 3.8 and 3.8
// ms on the long reads, 5.1, 4.9, 4.8 and 4.7 ms on the short ones; on 300 K
// windows all of them take the same.
void supermer_shape(int mode, int m, bool lexical, uint32_t n_buckets, uint64_t n_tiles, int num_sms, int* warps,
                    uint32_t* grid) {
    const uint64_t per_sm = (n_tiles + num_sms - 1) / num_sms;
    *warps = (int)(per_sm < 4 ? 4 : per_sm > SM_CTA_WARPS ? SM_CTA_WARPS : per_sm);
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, walk_kernel(mode, m, lexical, true, false), *warps * 32,
                                                      supermer_smem_bytes(mode, n_buckets, *warps)) != cudaSuccess)
        n = 1;
    if (n < 1) n = 1;
    const uint64_t want = (n_tiles + *warps - 1) / *warps, most = (uint64_t)num_sms * n;
    *grid = (uint32_t)(want < 1 ? 1 : want < most ? want : most);
}

// A record's nb bases (left aligned, the rest 0) or their reverse complement,
// whichever is smaller: the supermers of one locus on both strands then have
// one record.  (The k-mers are the same: they are canonical.)
template <int RW>
__device__ __forceinline__ void one_strand(u64 (&r)[RW], int nb) {
    constexpr int NW = 2 * RW;
    uint32_t x[NW + 1];  // the whole words reversed and complemented, then shifted left
#pragma unroll
    for (int i = 0; i < RW; ++i) {
        x[2 * i] = revcomp32((uint32_t)r[RW - 1 - i]);
        x[2 * i + 1] = revcomp32((uint32_t)(r[RW - 1 - i] >> 32));
    }
    x[NW] = 0;
    const uint32_t s = 64 * RW - 2 * nb;  // bits of the shift, < 64 RW
#pragma unroll
    for (int d = NW / 2; d > 0; d /= 2)
        if ((s >> 5) & d) {
#pragma unroll
            for (int i = 0; i < NW; ++i) x[i] = i + d < NW ? x[i + d < NW ? i + d : 0] : 0u;
        }
    u64 c[RW];
    bool less = false, same = true;
#pragma unroll
    for (int i = 0; i < RW; ++i) {
        c[i] = ((u64)__funnelshift_l(x[2 * i + 1], x[2 * i], s & 31) << 32) |
               __funnelshift_l(x[2 * i + 2], x[2 * i + 1], s & 31);
        less = less || (same && c[i] < r[i]);
        same = same && c[i] == r[i];
    }
    if (less) {
#pragma unroll
        for (int i = 0; i < RW; ++i) r[i] = c[i];
    }
}

// ---------------------------------------------------------------------------
// records from descriptors
// ---------------------------------------------------------------------------
// A slot in the supermer's bucket from the bucket's cursor, the record's
// bases gathered from the packed reads (the descriptors of a warp come from
// one tile, so these reads hit L1/L2).
//
// FINE: straight into the fine partitions, whose cursors start at their first
// record.  The records of a partition arrive one by one, but the partitions'
// open sectors (1 M x 32 bytes) stay in L2, so they leave it whole.  What
// bounds it is L2 requests: one atomic and one write per record, at random.
// Scattering into the buckets (4.4 and 3.8 ms; 5.9 and 4.4 with the
// sub-partition beside each record) and from there into the partitions (2.1 and
// 1.3 ms) took 8.0 and 5.7 ms on the long- and short-read workloads; this takes
// 4.0 and 3.3 (and 0.1 of the walk, which counts records per partition).
//
// SMs differ in how far the cursors and lines they need are, so every CTA takes
// its few descriptors and is done, and the next one goes where there is room:
// with 8 looping CTAs per SM some SMs were idle for the last fifth (4.5 and 3.9
// ms).  Few records in flight keep the open sectors few: descriptors a thread
// takes at a time, in CTAs of 512: 16-byte records 1 4.0 ms, 2 4.0, 3 4.1, 8 4.7;
// 32-byte records 3 3.6 ms, 4 3.4, 5 3.25, 6 3.25 (whose registers let fewer
// threads run); a tile's words are loaded before the slots are waited for.
constexpr int SD_NT = 512, SD_NARROW = 1, SD_WIDE = 5;  // threads a CTA, descriptors a thread
template <bool WIDE, bool FINE>
__global__ void __launch_bounds__(SD_NT) k_scatter_desc(const u64* __restrict__ desc, u64 n_desc,
                                                      const u64* __restrict__ packed, int k,
                                                      const u64* __restrict__ bucket_off, uint32_t* cursor,
                                                      unsigned long long* part_cursor, int sub_bits,
                                                      u64* __restrict__ records, u64 n_records, int* err) {
    constexpr int SD = WIDE ? SD_WIDE : SD_NARROW;
    constexpr int RW = WIDE ? 4 : 2;
    const u64 i0 = (u64)blockIdx.x * blockDim.x * SD + threadIdx.x;
    u64 dd[SD], slot[SD], w[SD][RW + 1];
#pragma unroll
    for (int j = 0; j < SD; ++j) {
        const u64 i = i0 + (u64)j * blockDim.x;
        dd[j] = i < n_desc ? __ldcs(desc + i) : ~0ULL;
    }
#pragma unroll
    for (int j = 0; j < SD; ++j) {
        slot[j] = ~0ULL;
        if (dd[j] != ~0ULL) {
            if constexpr (FINE) {
                const uint32_t b = (uint32_t)(dd[j] >> 43) & 0x1FFFu, sub = (uint32_t)(dd[j] >> 56);
                slot[j] = atomicAdd(part_cursor + ((b << sub_bits) | sub), 1ULL);
            } else {
                const uint32_t b = (uint32_t)(dd[j] >> 48);
                slot[j] = bucket_off[b] + atomicAdd(cursor + (size_t)b * SCATTER_CURSOR_STRIDE, 1u);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < SD; ++j) {  // up to RW words past the bases: the stream is padded
        const u64 pos = dd[j] == ~0ULL ? 0 : dd[j] & (FINE ? (1ULL << 36) - 1 : (1ULL << 40) - 1);
#pragma unroll
        for (int q = 0; q <= RW; ++q) w[j][q] = packed[(pos >> 5) + q];
    }
#pragma unroll
    for (int j = 0; j < SD; ++j) {
        const u64 d = dd[j];
        if (d == ~0ULL) continue;
        const uint32_t n = FINE ? (uint32_t)(d >> 36) & 0x7F : (uint32_t)(d >> 40) & 0xFF;
        const int nb = (int)n + k - 1;  // bases in the record
        const uint32_t off = 2 * ((uint32_t)d & 31u);
        u64 r[RW];
#pragma unroll
        for (int q = 0; q < RW; ++q) r[q] = keep_bases(funnel64(w[j][q], w[j][q + 1], off), nb - 32 * q);
        if (FINE) one_strand<RW>(r, nb);
        r[RW - 1] |= (u64)n;
        if (slot[j] >= n_records || (!FINE && slot[j] >= bucket_off[(uint32_t)(d >> 48) + 1])) {
            raise_error(err, HSK_DERR_BOUNDS);
            continue;
        }
        ulonglong2* dst = reinterpret_cast<ulonglong2*>(records) + (RW / 2) * slot[j];
#pragma unroll
        for (int q = 0; q < RW / 2; ++q) dst[q] = make_ulonglong2(r[2 * q], r[2 * q + 1]);
    }
}

void launch_scatter_desc(const uint64_t* desc, uint64_t n_desc, const uint64_t* packed, int k,
                         const uint64_t* bucket_off, uint32_t* cursor, uint64_t* part_cursor, int sub_bits,
                         uint64_t* records, uint64_t n_records, int* err, cudaStream_t st) {
    if (n_desc == 0) return;
    count_launch();
    const uint64_t per = SD_NT * (k <= 32 ? SD_NARROW : SD_WIDE), g = (n_desc + per - 1) / per;
    auto go = [&](auto kern) {
        kern<<<(unsigned)g, SD_NT, 0, st>>>((const u64*)desc, n_desc, (const u64*)packed, k, (const u64*)bucket_off, cursor,
                                (unsigned long long*)part_cursor, sub_bits, (u64*)records, n_records, err);
    };
    if (part_cursor) {
        if (k <= 32) go(k_scatter_desc<false, true>);
        else go(k_scatter_desc<true, true>);
    } else {
        if (k <= 32) go(k_scatter_desc<false, false>);
        else go(k_scatter_desc<true, false>);
    }
}

// ---------------------------------------------------------------------------
// exclusive scan of uint32 counts -> uint64 offsets (decoupled look-back)
// ---------------------------------------------------------------------------
constexpr int SCAN_ITEMS = 16;
constexpr int SCAN_TILE = 256 * SCAN_ITEMS;

uint64_t scan_status_words(uint64_t n) { return ((n + SCAN_TILE - 1) / SCAN_TILE + 1) * LB_PAD; }

// Also, when asked: a second copy of the offsets (cursors), and every
// 2^bnd_bits-th offset and the total (bnd).
__global__ void __launch_bounds__(256) k_scan_u32(const uint32_t* __restrict__ in, uint64_t n,
                                                  u64* __restrict__ out, u64* __restrict__ copy,
                                                  u64* __restrict__ bnd, int bnd_bits, u64* status,
                                                  uint32_t* tile_ctr, uint32_t epoch, int* err) {
    __shared__ uint32_t s_tile;
    __shared__ u64 s_scr[9];
    __shared__ u64 s_prefix;
    if (threadIdx.x == 0) s_tile = atomicAdd(tile_ctr, 1u);
    __syncthreads();
    const u64 tile = s_tile;
    const u64 base = tile * SCAN_TILE + (u64)threadIdx.x * SCAN_ITEMS;
    uint32_t v[SCAN_ITEMS];
    u64 sum = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        v[i] = base + i < n ? in[base + i] : 0u;
        sum += v[i];
    }
    u64 total;
    u64 excl = block_excl_sum<256, u64>(sum, s_scr, total);
    if (threadIdx.x == 0) {
        u64 pre = 0;
        if (tile == 0) {
            st_relaxed(status, lb_word(LB_PREFIX, epoch, total));
        } else {
            st_relaxed(status + tile * LB_PAD, lb_word(LB_AGG, epoch, total));
            pre = lookback_exclusive_win<16>(status, LB_PAD, tile, epoch, err);
            st_relaxed(status + tile * LB_PAD, lb_word(LB_PREFIX, epoch, pre + total));
        }
        s_prefix = pre;
    }
    __syncthreads();
    u64 run = s_prefix + excl;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const u64 at = base + i;
        if (at < n) {
            out[at] = run;
            if (copy) copy[at] = run;
            if (bnd && (at & ((1ULL << bnd_bits) - 1)) == 0) bnd[at >> bnd_bits] = run;
        }
        run += v[i];
    }
    if (base < n && base + SCAN_ITEMS >= n) {  // total
        out[n] = run;
        if (bnd) bnd[(n + (1ULL << bnd_bits) - 1) >> bnd_bits] = run;
    }
}

void launch_scan_u32(const uint32_t* in, uint64_t n, uint64_t* out, uint64_t* status,
                     uint32_t* tile_ctr, uint32_t epoch, int* err, cudaStream_t st, uint64_t* copy, uint64_t* bnd,
                     int bnd_bits) {
    if (n == 0) {
        cudaMemsetAsync(out, 0, sizeof(uint64_t), st);
        return;
    }
    uint64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    count_launch();
    k_scan_u32<<<(unsigned)tiles, 256, 0, st>>>(in, n, (u64*)out, (u64*)copy, (u64*)bnd, bnd_bits, (u64*)status,
                                                tile_ctr, epoch, err);
}

}  // namespace hsk
