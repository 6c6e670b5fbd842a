// encode_kernels.cuh -- CRC + polar encoder (Sec. II, x = u G) and the seeded workload
// generator (payload bits and BPSK-AWGN channel LLRs from Philox4x32-10).
#pragma once

#include "polar_common.cuh"

namespace polar {

// Encoder.  A frame's N / 32 code words sit on W = min(32, N / 32) lanes, H = N / 1024 (at least 1)
// words per lane, so a warp encodes 32 / W frames at once and loops over the batch; everything that
// depends on the code alone is prepared once per warp (expansion masks) or CTA (CRC table).
//   information word: the K information bits (payload, then CRC) are one bit string; word w of u holds
//     popcount(info mask of w) consecutive ones from the word's first information index on, spread
//     over the mask by five masked shifts (the expand of Warren, Hacker's Delight, sec. 7-5).
//   CRC: the remainder of payload(x) x^c is linear in the payload.  Each lane takes a 32-bit chunk and
//     looks its eight nibbles up in a shared table of their remainders (the XOR of the syndrome columns
//     of the bits set); the lanes' results are XORed.
//   transform: the Fig. 1 butterflies x_j ^= x_{j+d} (bit log2 d of j clear) -- in-word with shifts
//     for d < 32, across words with shuffles for 32 <= d < 1024 and within the lane for d >= 1024.
// What bounds it: instruction issue (about 200 per frame at N = 1024 against 190 bytes moved).  Measured
// at N = 1024, 10^5 frames: 29 us, against 280 us for a walk over the word's bits with a table lookup each.
constexpr int kEncWarps = 8;
__host__ __device__ inline int enc_chunks(int P) { return (P + 31) >> 5; }
// shared words: nibble table [8][16][chunks], then the payload chunks of each warp's frames
__host__ __device__ inline int enc_row_words(int N) { return N / 32 + 1; }
inline size_t enc_smem_bytes(int N, int P)
{
    const int frames = N >= 1024 ? 1 : 1024 / N;
    return 4 * ((size_t)128 * enc_chunks(P) + (size_t)kEncWarps * frames * enc_row_words(N));
}

template <int H>
__global__ void __launch_bounds__(kEncWarps * 32)
    encode_kernel(const DevCode* __restrict__ code, const uint8_t* __restrict__ payload, int B, int pay_bytes,
                  uint8_t* __restrict__ codeword)
{
    extern __shared__ uint32_t enc_smem[];
    const DevCode& C = *code;
    const int N = C.N, P = C.P, c = C.c, words = N >> 5, J = enc_chunks(P);
    const int W = min(words, 32), frames = 32 / W, rw = enc_row_words(N);
    const int lane = threadIdx.x & 31, wl = lane & (W - 1), slot = lane / W;
    uint32_t* table = enc_smem;
    uint32_t* row = enc_smem + 128 * J + ((threadIdx.x >> 5) * frames + slot) * rw;
    if (c > 0) {
        for (int q = threadIdx.x; q < 8 * J; q += blockDim.x) {
            const int j = q % J, nib = q / J;  // information indices 32 j + 4 nib ..
            uint32_t col[4], v[16];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = 32 * j + 4 * nib + i;
                col[i] = k < P ? C.colsyn[C.info_idx[k]] : 0u;
            }
            v[0] = 0u;
#pragma unroll
            for (int x = 1; x < 16; ++x) {
                const int top = x >= 8 ? 3 : x >= 4 ? 2 : x >= 2 ? 1 : 0;
                v[x] = v[x ^ (1 << top)] ^ col[top];
            }
#pragma unroll
            for (int x = 0; x < 16; ++x) table[(nib * 16 + x) * J + j] = v[x];
        }
    }
    // per word: information mask, its first information index, the five masks of the expansion
    uint32_t mask[H], mv[H][5];
    int k0[H];
    int before = 0;
#pragma unroll
    for (int h = 0; h < H; ++h) {
        uint32_t m = ~C.frozen_bits[wl + 32 * h];
        mask[h] = m;
        int sum = __popc(m);
        const int own = sum;
        for (int d = 1; d < W; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, sum, d, W);
            if (wl >= d) sum += o;
        }
        k0[h] = before + sum - own;
        before += __shfl_sync(0xffffffffu, sum, W - 1, W);
        uint32_t mk = ~m << 1;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            uint32_t mp = mk ^ (mk << 1);
            mp ^= mp << 2;
            mp ^= mp << 4;
            mp ^= mp << 8;
            mp ^= mp << 16;
            const uint32_t x = mp & m;
            mv[h][i] = x;
            m = (m ^ x) | (x >> (1 << i));
            mk &= ~mp;
        }
    }
    __syncthreads();
    // widest access every payload row allows: its start and length in bytes decide
    const int align = (int)((reinterpret_cast<uintptr_t>(payload) | (uintptr_t)pay_bytes) & 3u);
    // (unsigned: the last step of a grid may pass 2^31)
    const uint32_t frames_all = (uint32_t)B, stride = gridDim.x * kEncWarps * frames;
    for (uint32_t f0 = (blockIdx.x * kEncWarps + (threadIdx.x >> 5)) * frames; f0 < frames_all; f0 += stride) {
        const uint32_t frame = f0 + slot;
        const bool live = frame < frames_all;
        const uint8_t* pay = payload + (size_t)(live ? frame : f0) * pay_bytes;
        uint32_t crc = 0u;
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int j = wl + 32 * h;
            uint32_t x = 0u;
            if (j < J) {
                const int o = 4 * j;
                if (align == 0) {
                    x = *reinterpret_cast<const uint32_t*>(pay + o);
                } else if ((align & 1) == 0) {
                    x = *reinterpret_cast<const uint16_t*>(pay + o);
                    if (o + 2 < pay_bytes) x |= (uint32_t)*reinterpret_cast<const uint16_t*>(pay + o + 2) << 16;
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (o + i < pay_bytes) x |= (uint32_t)pay[o + i] << (8 * i);
                }
                if (P - 32 * j < 32) x &= (1u << (P - 32 * j)) - 1u;
                if (c > 0) {
#pragma unroll
                    for (int nib = 0; nib < 8; ++nib) crc ^= table[(nib * 16 + ((x >> (4 * nib)) & 15u)) * J + j];
                }
            }
            row[j] = x;  // chunks past the payload are 0
        }
        if (wl == 0) row[words] = 0u;
        if (W == 32) {
            crc = __reduce_xor_sync(0xffffffffu, crc);
        } else {
            for (int d = 1; d < W; d <<= 1) crc ^= __shfl_xor_sync(0xffffffffu, crc, d);
        }
        const uint32_t rc = c > 0 ? __brev(crc) >> (32 - c) : 0u;  // CRC bit string, MSB first
        __syncwarp();
        uint32_t w[H];
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int q = min(k0[h] >> 5, words - 1);  // (an all-frozen tail word has k0 = K, at most N)
            uint32_t x = __funnelshift_r(row[q], row[q + 1], k0[h] & 31);
            const int d = P - k0[h];  // the CRC starts d bits into this word's string
            if (d < 32) x |= d >= 0 ? rc << d : d > -32 ? rc >> -d : 0u;
#pragma unroll
            for (int i = 4; i >= 0; --i) x = (x & ~mv[h][i]) | ((x << (1 << i)) & mv[h][i]);
            w[h] = x & mask[h];
        }
        __syncwarp();  // the row is rewritten in the next round
        const uint32_t m[5] = {0x55555555u, 0x33333333u, 0x0F0F0F0Fu, 0x00FF00FFu, 0x0000FFFFu};
#pragma unroll
        for (int h = 0; h < H; ++h)
#pragma unroll
            for (int e = 0; e < 5; ++e) w[h] ^= (w[h] >> (1 << e)) & m[e];
        for (int D = 1; D < W; D <<= 1) {
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const uint32_t other = __shfl_xor_sync(0xffffffffu, w[h], D);
                if (!(lane & D)) w[h] ^= other;
            }
        }
#pragma unroll
        for (int hd = 1; hd < H; hd <<= 1)
#pragma unroll
            for (int h = 0; h < H; ++h)
                if (!(h & hd)) w[h] ^= w[h | hd];
        if (live) {
            uint32_t* out = reinterpret_cast<uint32_t*>(codeword + (size_t)frame * (N >> 3));
#pragma unroll
            for (int h = 0; h < H; ++h) out[wl + 32 * h] = w[h];
        }
    }
}

// ------------------------------------------------------------------------------ Philox4x32-10
struct U4 {
    uint32_t x, y, z, w;
};

// Round keys of a seed, made once on the host (kernel parameters: each round's key is an operand of its
// XOR and costs no instruction).
struct PhiloxKeys {
    uint32_t k[10][2];
};
inline PhiloxKeys philox_keys(uint64_t seed)
{
    PhiloxKeys r;
    uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    for (int i = 0; i < 10; ++i) {
        r.k[i][0] = k0;
        r.k[i][1] = k1;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return r;
}

__device__ __forceinline__ U4 philox4x32_10(U4 c, const PhiloxKeys& key)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c.x, p1 = (uint64_t)0xCD9E8D57u * c.z;
        c = U4{(uint32_t)(p1 >> 32) ^ c.y ^ key.k[r][0], (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ key.k[r][1], (uint32_t)p0};
    }
    return c;
}

// Payload rows: a CTA fills the bytes of kPayRows rows in shared memory, one Philox block (128 bits) per
// thread and step, and writes them out as one contiguous run in 16-byte stores.  (Rows are `bytes`
// long and start at any residue; stores from the block's thread went out in bytes or half words, 18 us
// per 10^5 rows of 62 bytes, now 7 us.)
constexpr int kPayRows = 64;
constexpr int kPayMaxBytes = 48 * 1024 / kPayRows;  // longer rows are written directly
__device__ __forceinline__ U4 payload_block(uint64_t f, int blk, const PhiloxKeys& key)
{
    return philox4x32_10(U4{(uint32_t)blk, (uint32_t)f, 0u, (uint32_t)(f >> 32)}, key);
}
// the block's bytes of a row of P bits (bytes = ceil(P / 8)); pad bits of the last byte are 0
__device__ __forceinline__ void payload_store(uint8_t* row, int blk, int P, int bytes, const U4& r)
{
    const uint32_t wv[4] = {r.x, r.y, r.z, r.w};
    uint8_t* p = row + 16 * blk;
    const uintptr_t at = reinterpret_cast<uintptr_t>(p);
    if (P - 128 * blk >= 128 && (at & 1u) == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if ((at & 3u) == 0) {
                reinterpret_cast<uint32_t*>(p)[q] = wv[q];
            } else {
                reinterpret_cast<uint16_t*>(p)[2 * q] = (uint16_t)wv[q];
                reinterpret_cast<uint16_t*>(p)[2 * q + 1] = (uint16_t)(wv[q] >> 16);
            }
        }
        return;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int by = 0; by < 4; ++by) {
            const int byte = (blk * 4 + q) * 4 + by;
            if (byte >= bytes) continue;
            uint8_t v = (uint8_t)(wv[q] >> (8 * by));
            const int valid = P - byte * 8;
            if (valid < 8) v &= (uint8_t)((1u << valid) - 1u);
            p[q * 4 + by] = v;
        }
    }
}
__global__ void __launch_bounds__(256)
    random_payload_kernel(int B, int P, const PhiloxKeys key, uint64_t frame0, uint8_t* __restrict__ out)
{
    extern __shared__ __align__(16) uint8_t pay_smem[];
    const int nblocks = (P + 127) >> 7, bytes = (P + 7) >> 3;
    const int row0 = blockIdx.x * kPayRows, rows = min(kPayRows, B - row0);
    for (int i = threadIdx.x; i < rows * nblocks; i += blockDim.x) {
        const int b = i / nblocks, blk = i % nblocks;
        payload_store(pay_smem + b * bytes, blk, P, bytes, payload_block(frame0 + (uint64_t)(row0 + b), blk, key));
    }
    __syncthreads();
    uint8_t* dst = out + (size_t)row0 * bytes;
    const int total = rows * bytes, vec = (reinterpret_cast<uintptr_t>(dst) & 15u) == 0 ? total >> 4 : 0;
    for (int i = threadIdx.x; i < vec; i += blockDim.x)
        reinterpret_cast<uint4*>(dst)[i] = reinterpret_cast<const uint4*>(pay_smem)[i];
    for (int i = 16 * vec + threadIdx.x; i < total; i += blockDim.x) dst[i] = pay_smem[i];
}
// Rows too long for shared memory: one thread per Philox block.
__global__ void random_payload_direct_kernel(int B, int P, const PhiloxKeys key, uint64_t frame0, uint8_t* __restrict__ out)
{
    const int nblocks = (int)(((long long)P + 127) >> 7), bytes = (int)(((long long)P + 7) >> 3);
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (long long)B * nblocks) return;
    const int b = (int)(gid / nblocks), blk = (int)(gid % nblocks);
    payload_store(out + (size_t)b * bytes, blk, P, bytes, payload_block(frame0 + (uint64_t)b, blk, key));
}

// One thread per Philox block (4 nodes) of one frame: Box-Muller on (w0, w1) and (w2, w3).  Bound by
// instruction issue (ten Philox rounds, two logarithms, square roots and sine / cosine pairs per 16
// bytes written).  N = 2^log2n, so frame and block come from shifts, and 2 / sigma^2 of a common sigma
// (scale_all) from the host: with a 64-bit division and a float division per thread 10^5 frames of
// N = 1024 took 260 us, without 232, and with the round keys as kernel parameters 223.
__global__ void awgn_llr_kernel(const uint8_t* __restrict__ codeword, int B, int log2n, float sigma_all, float scale_all,
                                const float* __restrict__ sigmas, const PhiloxKeys key, uint64_t frame0,
                                float* __restrict__ llr)
{
    const int N = 1 << log2n;
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (long long)B << (log2n - 2)) return;
    const int b = (int)(gid >> (log2n - 2)), blk = (int)gid & ((N >> 2) - 1);
    float sigma = sigma_all, scale = scale_all;
    if (sigmas) {
        sigma = sigmas[b];
        scale = 2.0f / (sigma * sigma);
    }
    const uint64_t f = frame0 + (uint64_t)b;
    const U4 r = philox4x32_10(U4{(uint32_t)blk, (uint32_t)f, 1u, (uint32_t)(f >> 32)}, key);
    const uint32_t e[2] = {r.x, r.z}, o[2] = {r.y, r.w};
    const uint8_t xb = codeword[(size_t)b * (N >> 3) + (blk >> 1)] >> ((blk & 1) * 4);
    float4 v;
    float* vp = &v.x;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const float u1 = (float)((e[p] >> 8) + 1u) * (1.0f / 16777216.0f);
        const float u2 = (float)(o[p] >> 8) * (1.0f / 16777216.0f);
        const float rad = sqrtf(-2.0f * logf(u1));
        float sn, cs;
        sincospif(2.0f * u2, &sn, &cs);
        const float z[2] = {rad * cs, rad * sn};
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = 2 * p + q;
            const float s = ((xb >> i) & 1) ? -1.0f : 1.0f;
            vp[i] = scale * (s + sigma * z[q]);
        }
    }
    reinterpret_cast<float4*>(llr + (size_t)b * N)[blk] = v;
}

}  // namespace polar
