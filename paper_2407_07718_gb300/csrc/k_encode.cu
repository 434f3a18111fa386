// k_encode.cu -- stage S1: 2-bit encoding of reads (Sec. 2.2: sequences are
// encoded before they are parsed into k-mers).
//
// One thread turns 16 ASCII bytes into half a packed word (16 bases, first
// base most significant) and a quarter of an invalid-mask word, so that every
// load and store of a warp is one run of bytes.  The kernel is bound by HBM (1
// byte read and 0.375 bytes written per base) once the arithmetic is short:
// byte compares, each several instructions, kept the integer pipe 93 % busy and
// took 0.83 and 1.18 ms on 1.5 and 2.0 Gbases; this takes 0.42 and 0.64.
#include "hsk_device.cuh"

namespace hsk {

// 4 ASCII bytes (little-endian in x) -> their codes in 2 bits per byte (A 0x41
// -> 0, C 0x43 -> 1, G 0x47 -> 2, T 0x54 -> 3: ((c >> 2) ^ (c >> 1)) & 3), right
// for the four letters; diff has a non-zero byte for every other one.
__device__ __forceinline__ uint32_t codes4(uint32_t x, uint32_t& diff) {
    const uint32_t c = ((x >> 2) ^ (x >> 1)) & 0x03030303u;
    // the codes as the selectors of a byte permutation of "ACGT"
    const uint32_t sel = __byte_perm(c | (c >> 4), 0, 0x4420);
    diff = x ^ __byte_perm(0x54474341u, 0, sel);
    return c;
}
// Invalid nibble (first byte in bit 3) of a diff word; the codes of its bytes cleared.
__device__ __noinline__ uint32_t invalid4(uint32_t diff, uint32_t& c) {
    const uint32_t bad = __vcmpne4(diff, 0u);
    c &= ~bad;
    return ((bad & 1u) << 3) | (((bad >> 8) & 1u) << 2) | (((bad >> 16) & 1u) << 1) | ((bad >> 24) & 1u);
}

// Units of 16 bases [u0, u1); n_bases bytes, the units past them invalid.  Unit
// u is the upper (u even) or lower half of packed word u / 2, and 16 bits of
// mask word u / 4, first bases uppermost.
__global__ void __launch_bounds__(256) k_encode(const char* __restrict__ reads, uint64_t n_bases,
                                                uint32_t* __restrict__ packed, uint16_t* __restrict__ invalid,
                                                uint64_t n_packed_words, uint64_t u0, uint64_t u1, bool aligned16) {
    constexpr int PER = 4;  // units a thread, a block apart
    const uint64_t first = u0 + (uint64_t)blockIdx.x * (256 * PER) + threadIdx.x;
    uint4 x[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const uint64_t u = first + (uint64_t)i * 256, b0 = u * 16;
        x[i] = make_uint4(0, 0, 0, 0);
        if (u >= u1) continue;
        if (aligned16 && b0 + 16 <= n_bases) {
            x[i] = __ldcs(reinterpret_cast<const uint4*>(reads + b0));  // streamed once: do not keep in L1/L2
        } else {
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                w[j] = 0;
                for (int b = 0; b < 4; ++b) {
                    const uint64_t g = b0 + 4 * j + b;
                    // bytes past the data read as 0 -> invalid
                    const uint32_t c = g < n_bases ? (uint32_t)(unsigned char)reads[g] : 0u;
                    w[j] |= c << (8 * b);
                }
            }
            x[i] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const uint64_t u = first + (uint64_t)i * 256;
        if (u >= u1) continue;
        const uint32_t w[4] = {x[i].x, x[i].y, x[i].z, x[i].w};
        uint32_t c[4], diff[4], bad = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) c[j] = codes4(w[j], diff[j]);
        if (diff[0] | diff[1] | diff[2] | diff[3]) {  // rare
#pragma unroll
            for (int j = 0; j < 4; ++j) bad |= invalid4(diff[j], c[j]) << (12 - 4 * j);
        }
        // four 2-bit codes, a byte apart, to the top byte of a product (no carries reach it)
        uint32_t code = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) code |= (c[j] * 0x40100401u) >> 24 << (24 - 8 * j);
        if (u / 2 < n_packed_words) packed[u ^ 1] = code;
        invalid[u ^ 3] = (uint16_t)bad;
    }
}

// Marks the first base of every non-empty read and checks the offsets:
// offsets[0] = 0, offsets[n_reads] = n_bases, non-decreasing.
__global__ void k_mark_starts(const uint64_t* __restrict__ offsets, uint64_t n_reads,
                              uint64_t n_bases, u64* __restrict__ start, int* err) {
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_reads) return;
    uint64_t s = offsets[i], e = offsets[i + 1];
    if (e < s || e > n_bases || (i == 0 && s != 0) || (i + 1 == n_reads && e != n_bases)) {
        raise_error(err, HSK_DERR_OFFSETS);
        return;
    }
    if (e > s) atomicOr(start + (s >> 6), 1ULL << (63 - (s & 63)));
}

// Packed sets: set y's reads are offsets[off0[y] .. off0[y] + n_reads[y]]
// (its own offsets, starting at 0) placed at base[y] of the packed bases;
// the bytes from the set's last base to base[y + 1] are padding and are set
// to 0 here (an invalid byte, so no window reaches into them).  Marks the first
// base of every non-empty read; offsets that leave the set's range are an
// error.
__global__ void k_mark_starts_sets(const uint64_t* __restrict__ offsets, const uint64_t* __restrict__ off0,
                                   const uint64_t* __restrict__ n_reads, const uint64_t* __restrict__ base,
                                   char* reads, u64* __restrict__ start, int* err) {
    const uint32_t y = blockIdx.y;
    const uint64_t nr = n_reads[y], b0 = base[y], b1 = base[y + 1];
    const uint64_t* o = offsets + off0[y];
    const uint64_t nb = o[nr];
    if (o[0] != 0 || b0 + nb > b1) {  // every block checks: nothing is written outside the set
        if (blockIdx.x == 0 && threadIdx.x == 0) raise_error(err, HSK_DERR_OFFSETS);
        return;
    }
    if (blockIdx.x == 0)
        for (uint64_t p = b0 + nb + threadIdx.x; p < b1; p += blockDim.x) reads[p] = 0;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nr; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t a = o[i], e = o[i + 1];
        if (e < a || e > nb) {
            raise_error(err, HSK_DERR_OFFSETS);
            return;
        }
        if (e > a) atomicOr(start + ((b0 + a) >> 6), 1ULL << (63 - ((b0 + a) & 63)));
    }
}

// Zero-fills up to ZERO_MAX regions in one launch (block row y: region y).
__global__ void __launch_bounds__(256) k_zero(const __grid_constant__ ZeroList L) {
    uint32_t* p = (uint32_t*)L.p[blockIdx.y];
    const uint64_t n = L.words[blockIdx.y];
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (uint64_t)gridDim.x * 256) p[i] = 0;
}

void launch_zero(const ZeroList& L, cudaStream_t st) {
    if (L.n == 0) return;
    uint64_t most = 0;
    for (int i = 0; i < L.n; ++i) most = L.words[i] > most ? L.words[i] : most;
    count_launch();
    const uint64_t bx = (most + 1023) / 1024;
    k_zero<<<dim3((unsigned)(bx < 1 ? 1 : bx > 256 ? 256 : bx), (unsigned)L.n), 256, 0, st>>>(L);
}

void launch_mark_starts_sets(const uint64_t* offsets, const uint64_t* off0, const uint64_t* n_reads,
                             const uint64_t* base, uint32_t n_sets, uint64_t max_reads, char* reads,
                             uint64_t* start_mask, int* err, cudaStream_t st) {
    if (n_sets == 0) return;
    count_launch();
    uint64_t bx = (max_reads + 255) / 256;
    if (bx < 1) bx = 1;
    if (bx > 1024) bx = 1024;
    k_mark_starts_sets<<<dim3((unsigned)bx, n_sets), 256, 0, st>>>(offsets, off0, n_reads, base, reads,
                                                                   (u64*)start_mask, err);
}

// bases [b0, b1), b0 a multiple of 64; whole mask words are written
static void encode_units(const char* reads, uint64_t n_bases, uint64_t b0, uint64_t b1, uint64_t* packed,
                         uint64_t* invalid, uint64_t n_packed_words, cudaStream_t st) {
    const uint64_t u0 = b0 / 64 * 4, u1 = (b1 + 63) / 64 * 4;
    if (u1 <= u0) return;
    count_launch();
    const bool al = (reinterpret_cast<uintptr_t>(reads) & 15) == 0;
    k_encode<<<(unsigned)((u1 - u0 + 1023) / 1024), 256, 0, st>>>(reads, n_bases, (uint32_t*)packed,
                                                                  (uint16_t*)invalid, n_packed_words, u0, u1, al);
}

void launch_encode(const char* reads, uint64_t n_bases, uint64_t* packed, uint64_t* invalid,
                   uint64_t n_packed_words, uint64_t n_mask_words, cudaStream_t st) {
    (void)n_mask_words;
    encode_units(reads, n_bases, 0, n_bases, packed, invalid, n_packed_words, st);
}

void launch_encode_range(const char* reads, uint64_t n_bases, uint64_t b0, uint64_t b1, uint64_t* packed,
                         uint64_t* invalid, uint64_t n_packed_words, cudaStream_t st) {
    encode_units(reads, n_bases, b0, b1, packed, invalid, n_packed_words, st);
}

void launch_mark_starts(const uint64_t* offsets, uint64_t n_reads, uint64_t n_bases,
                        uint64_t* start_mask, int* err, cudaStream_t st) {
    if (n_reads == 0) return;
    count_launch();
    k_mark_starts<<<(unsigned)((n_reads + 255) / 256), 256, 0, st>>>(offsets, n_reads, n_bases,
                                                                     (u64*)start_mask, err);
}

}  // namespace hsk
