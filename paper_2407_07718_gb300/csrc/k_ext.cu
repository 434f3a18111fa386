// k_ext.cu -- extension information of the kept k-mers (Sec. 3.3.2): the
// read and position of every occurrence of every k-mer the filter kept.
//
// After a count, the kept k-mers are sorted and distinct.  They are entered
// into a table of indices (open addressing over 32-bit slots holding index + 1
// and, above it, more hash bits, so one 32-bit compare-and-swap claims a slot
// whatever the key width).  A scan over every window then looks its canonical
// key up and, when the key is kept, emits the composite (k-mer index, global
// window start).  Sorting the composites (the LSD radix sort of k_sort.cu)
// puts each k-mer's occurrences together in position order, which is (read,
// position) order; a last pass turns the global start into (read, position in
// read) with a binary search over the read offsets.
//
// The payload codec (k_ext_encode / k_ext_decode) is the paper's encoding of
// extension information on its way to a destination: each item is
// (read, position); when both differ from the previous item of the stream by
// a value that fits an int8, the item is one flag byte plus the two int8
// differences, otherwise the flag byte plus the full uint32 read and uint32
// position.  Streams are cut into chunks of EXT_CHUNK items whose first item is
// always full, so chunks encode and decode independently.
#include "hsk_device.cuh"

namespace hsk {

// A slot of the table: the low idx_bits hold a kept k-mer's index + 1 (0: the
// slot is empty), the bits above some more hash bits of the k-mer, so that a
// probe reads the kept key only when it very likely matches.
struct ExtHash {
    uint32_t slot, tag;
};
__device__ __forceinline__ uint32_t ext_mix(uint32_t x) {
    x = (x ^ (x >> 16)) * 0x85EBCA6Bu;
    return x ^ (x >> 13);
}
__device__ __forceinline__ ExtHash ext_hash(uint32_t a, uint32_t b, uint32_t mask, int idx_bits) {
    ExtHash h;
    h.slot = ext_mix(a) & mask;
    h.tag = idx_bits < 32 ? ext_mix(b) << idx_bits : 0u;
    return h;
}
__device__ __forceinline__ ExtHash ext_hash(u64 k, uint32_t mask, int idx_bits) {
    const uint32_t l = (uint32_t)k, h = (uint32_t)(k >> 32);
    return ext_hash(l * 0x9E3779B1u + h * 0x85EBCA77u, l * 0xC2B2AE3Du + h * 0x27D4EB2Fu, mask, idx_bits);
}
__device__ __forceinline__ ExtHash ext_hash(const key128& k, uint32_t mask, int idx_bits) {
    const uint32_t a = (uint32_t)k.lo, b = (uint32_t)(k.lo >> 32), c = (uint32_t)k.hi, d = (uint32_t)(k.hi >> 32);
    return ext_hash(a * 0x9E3779B1u + b * 0x85EBCA77u + c * 0xC2B2AE3Du + d * 0x27D4EB2Fu,
                    a * 0x165667B1u + b * 0xD3A2646Du + c * 0xFD7046C5u + d * 0xB55A4F09u, mask, idx_bits);
}

template <typename K>
__global__ void __launch_bounds__(256) k_ext_insert(const K* __restrict__ keys, uint64_t n, uint32_t* table,
                                                    uint32_t mask, int idx_bits, int* err) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const ExtHash x = ext_hash(keys[i], mask, idx_bits);
        uint32_t h = x.slot;
        for (uint32_t probe = 0;; ++probe) {
            if (probe > mask) {  // never: the table has twice as many slots as keys
                raise_error(err, HSK_DERR_BOUNDS);
                break;
            }
            if (atomicCAS(&table[h], 0u, x.tag | ((uint32_t)i + 1)) == 0u) break;
            h = (h + 1) & mask;
        }
    }
}

// Index of `key` among the kept keys, or -1.
template <typename K>
__device__ __forceinline__ int64_t ext_find(const K& key, const K* __restrict__ kept, const uint32_t* __restrict__ table,
                                            uint32_t mask, int idx_bits) {
    const ExtHash x = ext_hash(key, mask, idx_bits);
    const uint32_t idx = idx_bits < 32 ? (1u << idx_bits) - 1u : 0xFFFFFFFFu;
    uint32_t h = x.slot;
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        const uint32_t v = table[h];
        if (v == 0) return -1;
        if ((v & ~idx) == x.tag && key_eq(kept[(v & idx) - 1], key)) return (int64_t)((v & idx) - 1);
        h = (h + 1) & mask;
    }
    return -1;
}

// A warp takes 1024 window starts, lane l the 32 that start in its word of
// packed bases: their validity from the invalid and read-start masks, their
// canonical keys rolled 16 at a time (KmerRoll), each valid one looked up.
// Kept ones emit (index << pos_bits) | start, buffered per warp and written
// with one atomic a buffer (128-bit composites when the two do not fit 64).
// Bound by the table's random reads (from L2 while it fits): 1.9 ms for 150 M
// windows and 3.6 M kept k-mers.  One thread per 64 windows, each window's key
// cut out and compared with a kept key at every probe, the masks shifted k
// times and one atomic a hit, took 7.4 ms.
constexpr int EXT_BUF = 128;  // composites buffered per warp
template <typename K>
__global__ void __launch_bounds__(256) k_ext_scan(const u64* __restrict__ packed, const u64* __restrict__ invalid,
                                                  const u64* __restrict__ start, uint64_t n_bases, int k,
                                                  const K* __restrict__ kept, const uint32_t* __restrict__ table,
                                                  uint32_t mask, int idx_bits, int pos_bits, bool wide_out, void* out,
                                                  uint64_t out_cap, unsigned long long* cursor, int* err) {
    constexpr bool WIDE = sizeof(K) == 16;
    __shared__ uint64_t s_pos[8][EXT_BUF];
    __shared__ uint32_t s_idx[8][EXT_BUF];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t n_pw = (n_bases + 31) / 32, n_mw = (n_bases + 63) / 64, tiles = (n_bases + 1023) / 1024;
    const u64 code = ~0ULL << (WIDE ? 128 - 2 * k : 64 - 2 * k);
    int nbuf = 0;  // composites buffered by this warp
    auto flush = [&]() {
        unsigned long long base = 0;
        __syncwarp();
        if (lane == 0) base = atomicAdd(cursor, (unsigned long long)nbuf);
        base = __shfl_sync(0xffffffffu, base, 0);
        for (int i = lane; i < nbuf; i += 32) {
            const uint64_t at = base + i, p = s_pos[warp][i];
            const u64 idx = s_idx[warp][i];
            if (at >= out_cap) {
                raise_error(err, HSK_DERR_BOUNDS);
            } else if (!wide_out) {
                reinterpret_cast<u64*>(out)[at] = (idx << pos_bits) | p;
            } else {
                key128 c;
                c.lo = p | (idx << pos_bits);
                c.hi = idx >> (64 - pos_bits);
                reinterpret_cast<key128*>(out)[at] = c;
            }
        }
        __syncwarp();
        nbuf = 0;
    };
    for (uint64_t t = (uint64_t)blockIdx.x * 8 + warp; t < tiles; t += (uint64_t)gridDim.x * 8) {
        const uint64_t p0 = t * 1024 + 32 * lane, wi = p0 >> 5, q = p0 >> 6;
        // window starts whose k bases are all valid and in one read, window j at bit j
        uint32_t V;
        {
            u64 iv[2], rs[3];
#pragma unroll
            for (int i = 0; i < 2; ++i) iv[i] = q + i < n_mw ? invalid[q + i] : ~0ULL;
#pragma unroll
            for (int i = 0; i < 3; ++i) rs[i] = q + i < n_mw ? start[q + i] : 0ULL;
            u64 bad = window_or64(iv[0], iv[1], k);
            if (k > 1) bad |= window_or64((rs[0] << 1) | (rs[1] >> 63), (rs[1] << 1) | (rs[2] >> 63), k - 1);
            V = ~__brev(lane & 1 ? (uint32_t)bad : (uint32_t)(bad >> 32));
            const uint64_t left = n_bases + 1 > p0 + k ? n_bases + 1 - (p0 + k) : 0;
            if (left < 32) V &= (1u << left) - 1u;
        }
        uint32_t w[6];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const u64 x = (i < 2 || WIDE) && wi + i < n_pw ? packed[wi + i] : 0ULL;
            w[2 * i] = (uint32_t)(x >> 32);
            w[2 * i + 1] = (uint32_t)x;
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            KmerRoll<WIDE> S;
            S.start(w + s, k);
            for (int j = 0; j < 16; ++j) {
                int64_t idx = -1;
                if ((V >> (16 * s + j)) & 1u) idx = ext_find(right_aligned(S.left(code), k), kept, table, mask, idx_bits);
                S.step();
                const uint32_t hit = __ballot_sync(0xffffffffu, idx >= 0);
                if (!hit) continue;
                if (idx >= 0) {
                    const int at = nbuf + __popc(hit & ((1u << lane) - 1u));
                    s_pos[warp][at] = p0 + 16 * s + j;
                    s_idx[warp][at] = (uint32_t)idx;
                }
                nbuf += __popc(hit);
                if (nbuf > EXT_BUF - 32) flush();
            }
        }
    }
    if (nbuf) flush();
}

// Sorted composites -> (read, position in read): read = the last read whose
// offset is <= the global start.
__global__ void __launch_bounds__(256) k_ext_decode_pos(const void* comp, bool wide, int pos_bits, uint64_t n,
                                                        const uint64_t* __restrict__ offsets, uint64_t n_reads,
                                                        uint32_t* __restrict__ occ_read, uint32_t* __restrict__ occ_pos) {
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (uint64_t)gridDim.x * blockDim.x) {
        const u64 c = wide ? reinterpret_cast<const key128*>(comp)[j].lo : reinterpret_cast<const u64*>(comp)[j];
        const u64 p = c & ((1ULL << pos_bits) - 1);
        uint64_t lo = 0, hi = n_reads;  // offsets[lo] <= p < offsets[hi]
        while (hi - lo > 1) {
            const uint64_t mid = (lo + hi) >> 1;
            if (offsets[mid] <= p) lo = mid;
            else hi = mid;
        }
        occ_read[j] = (uint32_t)lo;
        occ_pos[j] = (uint32_t)(p - offsets[lo]);
    }
}

void launch_ext_insert(const void* keys, int key_words, uint64_t n, uint32_t* table, uint32_t mask, int idx_bits,
                       int* err, cudaStream_t st) {
    if (n == 0) return;
    count_launch();
    const unsigned g = (unsigned)std::min<uint64_t>((n + 255) / 256, 65535);
    if (key_words == 1) k_ext_insert<u64><<<g, 256, 0, st>>>((const u64*)keys, n, table, mask, idx_bits, err);
    else k_ext_insert<key128><<<g, 256, 0, st>>>((const key128*)keys, n, table, mask, idx_bits, err);
}

void launch_ext_scan(const uint64_t* packed, const uint64_t* invalid, const uint64_t* start, uint64_t n_bases, int k,
                     const void* kept, const uint32_t* table, uint32_t mask, int idx_bits, int pos_bits, bool wide_out,
                     void* out, uint64_t out_cap, uint64_t* cursor, int* err, int grid, cudaStream_t st) {
    if (n_bases == 0) return;
    count_launch();
    const uint64_t tiles = (n_bases + 1023) / 1024;
    const unsigned g = (unsigned)std::min<uint64_t>((tiles + 7) / 8, (uint64_t)grid);
    if (k <= 32)
        k_ext_scan<u64><<<g, 256, 0, st>>>((const u64*)packed, (const u64*)invalid, (const u64*)start, n_bases, k,
                                           (const u64*)kept, table, mask, idx_bits, pos_bits, wide_out, out, out_cap,
                                           (unsigned long long*)cursor, err);
    else
        k_ext_scan<key128><<<g, 256, 0, st>>>((const u64*)packed, (const u64*)invalid, (const u64*)start, n_bases, k,
                                              (const key128*)kept, table, mask, idx_bits, pos_bits, wide_out, out,
                                              out_cap, (unsigned long long*)cursor, err);
}

void launch_ext_decode_pos(const void* comp, bool wide, int pos_bits, uint64_t n, const uint64_t* offsets,
                           uint64_t n_reads, uint32_t* occ_read, uint32_t* occ_pos, int grid, cudaStream_t st) {
    if (n == 0) return;
    count_launch();
    const unsigned g = (unsigned)std::min<uint64_t>((n + 255) / 256, (uint64_t)grid);
    k_ext_decode_pos<<<g, 256, 0, st>>>(comp, wide, pos_bits, n, offsets, n_reads, occ_read, occ_pos);
}

// ---------------------------------------------------------------------------
// the extension-information codec (Sec. 3.3.2)
// ---------------------------------------------------------------------------
// Item i of a stream: (read[i], pos[i]).  Flag byte: 1 = deltas follow (two
// int8: read - previous read, pos - previous pos), 0 = full values follow
// (uint32 read, uint32 pos, little endian).  The first item of every chunk of
// EXT_CHUNK items is full.  Sizes: 3 or 9 bytes.
constexpr uint32_t EXT_CHUNK = 1024;

__device__ __forceinline__ bool ext_small(uint32_t r, uint32_t p, uint32_t pr, uint32_t pp) {
    const long long dr = (long long)r - (long long)pr, dp = (long long)p - (long long)pp;
    return dr >= -128 && dr <= 127 && dp >= -128 && dp <= 127;
}

// bytes of item i (pass 1)
__global__ void k_ext_sizes(const uint32_t* __restrict__ rd, const uint32_t* __restrict__ ps, uint64_t n,
                            uint32_t* __restrict__ size) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const bool delta = (i % EXT_CHUNK) != 0 && ext_small(rd[i], ps[i], rd[i - 1], ps[i - 1]);
        size[i] = delta ? 3u : 9u;
    }
}

// item i written at byte off[i] (pass 2, off = exclusive scan of the sizes)
__global__ void k_ext_encode(const uint32_t* __restrict__ rd, const uint32_t* __restrict__ ps, uint64_t n,
                             const uint64_t* __restrict__ off, uint8_t* __restrict__ out) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        uint8_t* o = out + off[i];
        const bool delta = (i % EXT_CHUNK) != 0 && ext_small(rd[i], ps[i], rd[i - 1], ps[i - 1]);
        if (delta) {
            o[0] = 1;
            o[1] = (uint8_t)(int8_t)((long long)rd[i] - (long long)rd[i - 1]);
            o[2] = (uint8_t)(int8_t)((long long)ps[i] - (long long)ps[i - 1]);
        } else {
            o[0] = 0;
            for (int b = 0; b < 4; ++b) {
                o[1 + b] = (uint8_t)(rd[i] >> (8 * b));
                o[5 + b] = (uint8_t)(ps[i] >> (8 * b));
            }
        }
    }
}

// One thread per chunk: walk the chunk's items from its first (full) item.
__global__ void k_ext_decode(const uint8_t* __restrict__ in, uint64_t n_bytes, uint64_t n,
                             const uint64_t* __restrict__ chunk_off, uint32_t* __restrict__ rd,
                             uint32_t* __restrict__ ps, int* err) {
    const uint64_t chunks = (n + EXT_CHUNK - 1) / EXT_CHUNK;
    for (uint64_t c = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; c < chunks;
         c += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t at = chunk_off[c];
        uint32_t r = 0, p = 0;
        const uint64_t i1 = (c + 1) * EXT_CHUNK < n ? (c + 1) * EXT_CHUNK : n;
        for (uint64_t i = c * EXT_CHUNK; i < i1; ++i) {
            if (at >= n_bytes) {
                raise_error(err, HSK_DERR_BOUNDS);
                return;
            }
            const uint8_t f = in[at];
            if (f == 1 && i != c * EXT_CHUNK && at + 3 <= n_bytes) {
                r = (uint32_t)((long long)r + (int8_t)in[at + 1]);
                p = (uint32_t)((long long)p + (int8_t)in[at + 2]);
                at += 3;
            } else if (f == 0 && at + 9 <= n_bytes) {
                r = p = 0;
                for (int b = 0; b < 4; ++b) {
                    r |= (uint32_t)in[at + 1 + b] << (8 * b);
                    p |= (uint32_t)in[at + 5 + b] << (8 * b);
                }
                at += 9;
            } else {
                raise_error(err, HSK_DERR_BOUNDS);
                return;
            }
            rd[i] = r;
            ps[i] = p;
        }
    }
}

// byte offset of each chunk's first item (from the item offsets)
__global__ void k_ext_chunk_off(const uint64_t* __restrict__ off, uint64_t n, uint64_t* __restrict__ chunk_off) {
    const uint64_t chunks = (n + EXT_CHUNK - 1) / EXT_CHUNK;
    for (uint64_t c = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; c < chunks;
         c += (uint64_t)gridDim.x * blockDim.x)
        chunk_off[c] = off[c * EXT_CHUNK];
}

uint64_t ext_chunk_items() { return EXT_CHUNK; }

void launch_ext_sizes(const uint32_t* rd, const uint32_t* ps, uint64_t n, uint32_t* size, int grid, cudaStream_t st) {
    if (n == 0) return;
    count_launch();
    k_ext_sizes<<<(unsigned)std::min<uint64_t>((n + 255) / 256, (uint64_t)grid), 256, 0, st>>>(rd, ps, n, size);
}
void launch_ext_encode(const uint32_t* rd, const uint32_t* ps, uint64_t n, const uint64_t* off, uint8_t* out,
                       int grid, cudaStream_t st) {
    if (n == 0) return;
    count_launch();
    k_ext_encode<<<(unsigned)std::min<uint64_t>((n + 255) / 256, (uint64_t)grid), 256, 0, st>>>(rd, ps, n,
                                                                                              off, out);
}
void launch_ext_chunk_off(const uint64_t* off, uint64_t n, uint64_t* chunk_off, int grid, cudaStream_t st) {
    if (n == 0) return;
    count_launch();
    const uint64_t chunks = (n + EXT_CHUNK - 1) / EXT_CHUNK;
    const unsigned g = (unsigned)std::min<uint64_t>((chunks + 255) / 256, (uint64_t)grid);
    k_ext_chunk_off<<<g, 256, 0, st>>>(off, n, chunk_off);
}
void launch_ext_decode(const uint8_t* in, uint64_t n_bytes, uint64_t n, const uint64_t* chunk_off, uint32_t* rd,
                       uint32_t* ps, int* err, int grid, cudaStream_t st) {
    if (n == 0) return;
    count_launch();
    const uint64_t chunks = (n + EXT_CHUNK - 1) / EXT_CHUNK;
    const unsigned g = (unsigned)std::min<uint64_t>((chunks + 255) / 256, (uint64_t)grid);
    k_ext_decode<<<g, 256, 0, st>>>(in, n_bytes, n, chunk_off, rd, ps, err);
}

}  // namespace hsk
