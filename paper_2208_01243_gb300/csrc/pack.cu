// 2-bit packer: ASCII A/C/G/T -> 0/1/2/3, first base in the top two bits of each 64-bit word; sequences at any byte
// offset, word offsets given or i * stride.
//
// A warp takes a batch of up to 32 sequences, one per lane for their offsets and lengths, and walks the words of all
// of them as one list, a word per lane whatever the sequences' lengths (a scan over the batch gives each sequence's
// place, five shuffles find a word's sequence), so lanes stay busy over uneven reads and the offsets are read once,
// coalesced.  A lane reads its word's 32 bytes as two aligned 16-byte chunks, converts them as they lie (bytes outside
// the sequence read as 'A', code 0), takes the code bits of the next chunk from the next lane, and shifts the 96 bits
// by the sequence's offset inside its first chunk: the alignment costs two funnel shifts on codes instead of eight on
// bytes and nine 4-byte loads.  Each sequence has one item more than words, which only supplies that next chunk.
// Every chunk read holds a byte of its sequence, so no read crosses into another page.
//
// (c >> 1) & 3 maps A, C, T, G (0x41, 0x43, 0x54, 0x47) to 0, 1, 2, 3; a byte is one of the four exactly when it equals
// "ACTG" at that value, looked up for four bytes by one byte permute; one multiply lines the values up as the permute's
// selector, another gathers them into a byte, and one XOR over 16 bases turns 2 and 3 into the codes of T and G.
// Bytes next to a sequence are converted like its own: the shift drops those before it and a mask those after it;
// only a chunk that shows a byte other than the four is looked at again, with the bytes outside the sequence masked.
//
// What bounds it: the latency of the 16-byte loads (6.3 of 14 stalls an issue) and the integer pipe (59 % busy); 40 registers, for 48
// warps on an SM, measured better than more registers or loads issued a turn ahead (136 us with 55 registers, 132 us
// with the loads ahead).  1M sequences of 100-1,000 bp (391 MB) in 123 us, 4.2 TB/s of 6.8, from 901 us with a warp
// per sequence and a byte per lane; 1M of 150 bp 62 us (from 392 us; a thread per word in fixed slots 63 us, and 105
// us over uneven lengths against 54 us here).
#include <algorithm>

#include "aim_internal.cuh"

namespace aim {
namespace {

constexpr int kPackWarps = 8;   // per block

// four bytes (first in the low byte) -> (c >> 1) & 3 of each, the first's in the top two bits of the top byte; diff
// collects bytes that are none of the four letters
__device__ __forceinline__ uint32_t gather4(uint32_t x, uint32_t& diff) {
    const uint32_t y = (x >> 1) & 0x03030303u;
    const uint32_t sel = __byte_perm(y * 0x110u, 0u, 0x4431u);   // y_0 | y_1 << 4 in byte 1 of the product, y_2, y_3 in 3
    diff |= __byte_perm(0x47544341u, 0u, sel) ^ x;                // "ACTG"[y_k] against the byte
    return y * 0x40100401u;   // 2^30 + 2^20 + 2^10 + 1: no carries into the top byte
}

// 16 bytes -> 32 bits, first base on top; values of (c >> 1) & 3 (codes_of makes them codes)
__device__ __forceinline__ uint32_t gather16(uint4 u, uint32_t& diff) {
    const uint32_t a = gather4(u.x, diff), b = gather4(u.y, diff), c = gather4(u.z, diff), d = gather4(u.w, diff);
    return __byte_perm(__byte_perm(d, c, 0x0073u), __byte_perm(b, a, 0x0073u), 0x5410u);
}
__device__ __forceinline__ uint32_t codes_of(uint32_t z) { return z ^ ((z >> 1) & 0x55555555u); }

// the bytes of x that are A, C, G or T; the others as 'A'
__device__ __forceinline__ uint32_t letters_only(uint32_t x) {
    uint32_t r = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t c = (x >> (8 * k)) & 0xffu;
        r |= (c == 'C' || c == 'G' || c == 'T' ? c : (uint32_t)'A') << (8 * k);
    }
    return r;
}

// a chunk that showed some other byte: the bytes outside the sequence (not in m) count as 'A'; any left inside is
// bad, code 0
__device__ __noinline__ uint32_t gather16_checked(uint4 u, uint4 m, bool& bad) {
    auto keep = [](uint32_t k, uint32_t x) { return (x & k) | (0x41414141u & ~k); };
    u = make_uint4(keep(m.x, u.x), keep(m.y, u.y), keep(m.z, u.z), keep(m.w, u.w));
    uint32_t diff = 0;
    uint32_t z = gather16(u, diff);
    if (diff) {
        bad = true;
        z = gather16(make_uint4(letters_only(u.x), letters_only(u.y), letters_only(u.z), letters_only(u.w)), diff);
    }
    return z;
}

__device__ __forceinline__ uint32_t shr_clamp(uint32_t x, uint32_t s) {   // 0 for s >= 32
    uint32_t r;
    asm("shr.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
    return r;
}

// SHARED: `parts` warps share a batch (few sequences, which may be long), each taking every parts-th turn; batches are then
// one sequence, the grid covers them at once, and the parts lie in one block of WARPS warps, which gather its flag.  (With
// the flags zeroed by a memset before the launch 64 sequences of 150 bp took 6.2 us, 2.7 now.)
template <int WARPS, bool SHARED>
__global__ void __launch_bounds__(32 * WARPS, 48 / WARPS) pack_kernel(const uint8_t* __restrict__ ascii,
                                                               const uint64_t* __restrict__ char_off,
                                                               const uint32_t* __restrict__ len, uint32_t count,
                                                               uint32_t batch, uint32_t parts,
                                                               uint64_t* __restrict__ packed,
                                                               const uint64_t* __restrict__ word_off,
                                                               uint64_t word_stride, uint8_t* __restrict__ bad) {
    __shared__ uint4 s_first[17];   // [h]: ones in the first h bytes of a chunk
    __shared__ uint32_t s_bad[WARPS];   // SHARED: whether a warp saw a byte that is none of the four
    if (SHARED && threadIdx.x < WARPS) s_bad[threadIdx.x] = 0;
    if (threadIdx.x < 17) {
        auto word = [&](int q) -> uint32_t {
            const int h = (int)threadIdx.x - 4 * q;
            return h >= 4 ? 0xffffffffu : h <= 0 ? 0u : (1u << (8 * h)) - 1u;
        };
        s_first[threadIdx.x] = make_uint4(word(0), word(1), word(2), word(3));
    }
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint64_t nbatches = ((uint64_t)count + batch - 1) / batch;
    for (uint64_t work = warp; work < nbatches * parts; work += nwarps) {
        const uint32_t first = (uint32_t)(work / parts) * batch, part = (uint32_t)(work % parts);
        // this lane's sequence
        const bool have = lane < batch && lane < count - first;
        uint32_t L = 0, items = 0;
        uint64_t from = 0, to = 0;
        if (have) {
            const uint32_t i = first + lane;
            L = __ldg(len + i);
            from = reinterpret_cast<uint64_t>(ascii) + __ldg(char_off + i);
            to = word_off ? __ldg(word_off + i) : i * word_stride;
            const uint32_t nw = (L + 31) >> 5;
            const bool fits = word_off || nw <= word_stride;   // longer than the fixed slot: flag, write nothing
            items = fits && nw ? nw + 1 : 0;
            if (SHARED && !fits) s_bad[threadIdx.x >> 5] = 1;
            if (!SHARED && bad) bad[i] = !fits;
        }
        __syncwarp();   // bad[] starts at 0 before any lane sets it
        // all sequences at once, or one by one where the list's length might leave 32 bits (over 2 G bases in one)
        const bool huge = __any_sync(kFull, items > (1u << 26));
        for (uint32_t todo = __ballot_sync(kFull, items != 0); todo;) {
            const uint32_t take = huge ? todo & (0u - todo) : todo;
            todo &= ~take;
            const uint32_t mine = (take >> lane) & 1u ? items : 0u;
            uint32_t upto = mine;   // items of this and the sequences before it
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, upto, o);
                if ((int)lane >= o) upto += t;
            }
            const uint32_t total = __shfl_sync(kFull, upto, 31);
            const uint32_t before = upto - mine;
            // 31 items a turn; lane 31 only supplies the next chunk to lane 30
            for (uint32_t base = 31 * part; base < total; base += 31 * parts) {
                const uint32_t it = base + lane;
                uint32_t s = 0;   // sequences whose items all come before this one
#pragma unroll
                for (int step = 16; step > 0; step >>= 1)
                    if (__shfl_sync(kFull, upto, (int)(s + step - 1)) <= it) s += step;
                const uint32_t sL = __shfl_sync(kFull, L, s), w = it - __shfl_sync(kFull, before, s);
                const uint64_t sfrom = __shfl_sync(kFull, from, s), sto = __shfl_sync(kFull, to, s);
                const uint32_t phase = (uint32_t)sfrom & 15u, nw = (sL + 31) >> 5;
                // the sequence's bytes from this item's chunks on, counted from the chunk's start
                const int left = it >= total ? 0 : w + 2 < nw ? 64 : (int)(sL - 32 * w) + (int)phase;
                const uint4* src = reinterpret_cast<const uint4*>(sfrom & ~15ull) + 2ull * w;
                uint4 u0 = make_uint4(0x41414141u, 0x41414141u, 0x41414141u, 0x41414141u), u1 = u0;
                if (left > 0) u0 = __ldg(src);
                if (left > 16) u1 = __ldg(src + 1);
                bool b = false;
                uint32_t d0 = 0, d1 = 0;
                uint32_t z0 = gather16(u0, d0), z1 = gather16(u1, d1);
                if (d0 | d1) {
                    uint4 m = s_first[min(max(left, 0), 16)];
                    const uint4 l = s_first[w == 0 ? phase : 0u];
                    m = make_uint4(m.x & ~l.x, m.y & ~l.y, m.z & ~l.z, m.w & ~l.w);
                    z0 = gather16_checked(u0, m, b);
                    z1 = gather16_checked(u1, s_first[min(max(left - 16, 0), 16)], b);
                }
                const uint32_t z2 = __shfl_down_sync(kFull, z0, 1);
                if (lane < 31 && it < total && w < nw) {
                    const uint32_t nb = min(sL - 32 * w, 32u);   // bases of this word
                    const uint32_t hi = codes_of(__funnelshift_l(z1, z0, 2 * phase)) & ~shr_clamp(~0u, 2 * nb);
                    const uint32_t lo = codes_of(__funnelshift_l(z2, z1, 2 * phase)) &
                                        ~shr_clamp(~0u, 2 * max(nb, 16u) - 32);
                    packed[sto + w] = ((uint64_t)hi << 32) | lo;
                }
                if (bad && b) {
                    if (SHARED) s_bad[threadIdx.x >> 5] = 1;
                    else bad[first + s] = 1;
                }
            }
        }
    }
    if (SHARED && bad) {
        __syncthreads();
        const uint64_t i = (uint64_t)blockIdx.x * (WARPS / parts) + threadIdx.x;   // parts divides a block's warps
        if (threadIdx.x < WARPS / parts && i < count) {
            uint32_t any = 0;
            for (uint32_t k = 0; k < parts; ++k) any |= s_bad[threadIdx.x * parts + k];
            bad[i] = any != 0;
        }
    }
}

}  // namespace

cudaError_t launch_pack(const uint8_t* ascii, const uint64_t* char_off, const uint32_t* len, uint32_t count,
                        uint64_t* packed, const uint64_t* word_off, uint64_t word_stride, uint8_t* bad,
                        cudaStream_t st) {
    if (count == 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // batches of up to 32 sequences, smaller (and then shared by several warps) while that leaves SMs without 16 warps
    const uint32_t want = (uint32_t)sms * 16;
    uint32_t batch = 32, parts = 1;
    while (batch > 1 && ((uint64_t)count + batch - 1) / batch < want) batch /= 2;
    const uint64_t batches = ((uint64_t)count + batch - 1) / batch;
    // (no more than a slot's words keep busy, where slots are fixed: 61 pairs of 150 bp 28.7 us a call, 31.8 with 16)
    while (parts < 16 && batches * parts < want / 2 && (word_off || 31ull * parts <= word_stride)) parts *= 2;
    const uint64_t warps = batches * parts;
    const int per_block = std::max(kPackWarps, (int)parts);
    const uint64_t blocks = std::min<uint64_t>((warps + per_block - 1) / per_block, (uint64_t)sms * 32);
    auto kernel = parts == 1 ? pack_kernel<kPackWarps, false> : parts <= kPackWarps ? pack_kernel<kPackWarps, true> : pack_kernel<16, true>;
    kernel<<<(unsigned)blocks, 32 * per_block, 0, st>>>(ascii, char_off, len, count, batch, parts, packed, word_off,
                                                        word_stride, bad);
    return cudaGetLastError();
}

}  // namespace aim
