// pc_encode (Eq. 1 and the CRC of Sec. IV): payload bytes in, codeword bytes out.
//
// Bound by integer instruction issue (326 warp instructions a frame at N = 1024, the logic pipe at 79%
// of its rate; its HBM floor, K - r bytes read and N written, is half of its time).
// A codeword is N bits in 32-bit words, one word a lane (two at N = 2048), 32 * 32 / N frames to a
// warp, so the butterflies are shifts inside a word and shuffles between lanes and a warp's output
// is 1 KB of consecutive bytes, stored 16 bytes a lane.  The payload rows of a warp's frames are one
// run of bytes whatever K - r is: it is read 32 bytes a lane while the frames before are encoded,
// packed to a bit string in shared memory, and every later use (the payload words of the CRC, the
// information bits of a codeword word) is a 32-bit window of that string, so no row has to be
// aligned.  The CRC is the XOR of one table entry per four payload bits.
//
// 262,144 frames of N = 1024, K = 512 with CRC-24: 105 us, 3.8 TB/s (one CTA a frame on bytes in
// shared memory, with ten barriers a frame: 2,192 us).  Packing with byte dot products and the CRC's
// addresses by one logic operation each measured 124 us against 115 at the time, with 20 instructions fewer.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <memory>

#include "pcbp_internal.h"

namespace pcbp {

namespace {

template <int LOGN>
struct EncGeo {
    static constexpr int N = 1 << LOGN;
    static constexpr int W = N >= 32 ? N / 32 : 1;         // words of a codeword
    static constexpr int WPL = W > 32 ? W / 32 : 1;        // words per lane
    static constexpr int LPF = W / WPL;                    // lanes per frame
    static constexpr int FPW = 32 / LPF;                   // frames per warp
    static constexpr int UNIT = FPW * N;                   // codeword bits of a warp at a time
    // payload bits of a unit, up to 15 bits before them and the windows that run past them
    static constexpr int BIT_WORDS = (UNIT / 32 + 5 + 3) & ~3;
    static constexpr int LOADS = (UNIT / 32 + 1 + 31) / 32; // words of the string that a lane packs
    static constexpr int TABLE = 128 * W;                  // [nibble of the word][value][word]
    static constexpr int WARPS = 8;
    // word of contribution j while the table is made: a word in 33 left free, so that the lanes, 32
    // contributions apart, meet on no bank (one frame of N = 2048, K = 2047 23.1 -> 16.8 us, 49,157
    // frames of K = 2046 113 -> 78)
    __host__ __device__ static constexpr int padded(int j) { return j + (j >> 5); }
    static constexpr size_t smem(int K) { return 4 * (size_t(TABLE) + std::max(WARPS * BIT_WORDS, padded(K) + 1)); }
};

// 4 bytes (their lowest bits) to 4 bits, and back.
__device__ __forceinline__ uint32_t pack4(uint32_t b) { return ((b & 0x01010101u) * 0x01020408u) >> 24; }
__device__ __forceinline__ uint32_t spread4(uint32_t v) { return ((v & 15u) * 0x00204081u) & 0x01010101u; }

// WIDE: the codewords start on a 16-byte boundary and are stored 16 bytes a lane (8 below N = 32), else byte
// by byte.  A kernel for each: with both in one, the aligned stores of N = 128 and 256 were 5% slower.
template <int LOGN, bool WIDE>
__global__ void __launch_bounds__(256) encode_kernel(const __grid_constant__ EncParams P)
{
    using Geo = EncGeo<LOGN>;
    constexpr int N = Geo::N, W = Geo::W, WPL = Geo::WPL, LPF = Geo::LPF, FPW = Geo::FPW;
    extern __shared__ __align__(16) uint32_t s_enc[];
    uint32_t* const table = s_enc;
    uint32_t* const strings = s_enc + Geo::TABLE;       // a bit string per warp; the contributions while the table is made
    const int Kp = P.Kp, r = P.r;
    const int lane = int(threadIdx.x & 31), warp = int(threadIdx.x >> 5);
    if (r > 0) {
        for (int i = threadIdx.x; i < Kp; i += blockDim.x) strings[Geo::padded(i)] = P.crc_pay[i];
        __syncthreads();
        for (int i = threadIdx.x; i < Geo::TABLE; i += blockDim.x) {
            const int w = i % W, v = (i / W) & 15, k = i / (16 * W);
            uint32_t c = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int j = 32 * w + 4 * k + b;
                if (((v >> b) & 1) && j < Kp) c ^= strings[Geo::padded(j)];
            }
            table[i] = c;
        }
    }
    // the lane's codeword words: information positions, rank of the first, and the steps that move
    // the low bits of a word to those positions (each bit by a power of two, the largest first):
    // the expand operation of H. S. Warren, Hacker's Delight, section 7-5, its names kept (mk, mp, mv)
    const int w0 = lane % LPF;
    uint32_t info[WPL], step[WPL][5];
    int rank[WPL];
    {
        int before = 0;
#pragma unroll
        for (int q = 0; q < WPL; ++q) {
            const int w = w0 + 32 * q;
            const uint32_t all = N >= 32 ? 0xffffffffu : (1u << (N & 31)) - 1u;
            before = 0;
            for (int i = 0; i < w; ++i) before += __popc(~P.frozen[i]);
            rank[q] = before;
            uint32_t m = ~P.frozen[w] & all;
            info[q] = m;
            uint32_t mk = ~m << 1;                      // zeros to the right of a position, by parity
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                uint32_t mp = mk ^ (mk << 1);
                mp ^= mp << 2;
                mp ^= mp << 4;
                mp ^= mp << 8;
                mp ^= mp << 16;
                const uint32_t mv = mp & m;
                step[q][i] = mv;
                m = (m ^ mv) | (mv >> (1 << i));
                mk &= ~mp;
            }
        }
    }
    __syncthreads();                                    // the table is made
    uint32_t* const bits = strings + warp * Geo::BIT_WORDS;
    const uintptr_t begin = reinterpret_cast<uintptr_t>(P.payload), end = begin + size_t(P.B) * Kp;
    // the payload of a unit as a bit string, from the 16-byte boundary at or before it: 32 bytes a
    // lane and word, read while the unit before is encoded
    uint4 raw[Geo::LOADS][2];
    auto load = [&](uintptr_t from, int frames) {
        const uintptr_t base = from & ~uintptr_t(15);
        const int words = (int(from & 15u) + frames * Kp + 31) >> 5;
        const bool inside = base >= begin && base + 32 * size_t(words) <= end;
#pragma unroll
        for (int k = 0; k < Geo::LOADS; ++k) {
            const int i = lane + 32 * k;
            const uintptr_t p = base + 32 * size_t(i);
            if (inside) {
                if (i < words) {
                    raw[k][0] = __ldcs(reinterpret_cast<const uint4*>(p));
                    raw[k][1] = __ldcs(reinterpret_cast<const uint4*>(p) + 1);
                }
            } else {
                // the ends of the buffer: only its own bytes
                uint32_t w[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    w[q] = 0;
#pragma unroll 1
                    for (int b = 0; b < 4; ++b) {
                        const uintptr_t a = p + size_t(4 * q + b);
                        if (i < words && a >= begin && a < end) w[q] |= uint32_t(*reinterpret_cast<const uint8_t*>(a)) << (8 * b);
                    }
                }
                raw[k][0] = make_uint4(w[0], w[1], w[2], w[3]);
                raw[k][1] = make_uint4(w[4], w[5], w[6], w[7]);
            }
        }
    };
    // units of FPW frames, warp by warp over the grid
    const int64_t units = (P.B + FPW - 1) / FPW, stride = int64_t(gridDim.x) * Geo::WARPS;
    auto frames_of = [&](int64_t u) { return u + 1 < units ? FPW : int(P.B - u * FPW); };
    int64_t u = int64_t(blockIdx.x) * Geo::WARPS + warp;
    uintptr_t from = begin + size_t(u) * (FPW * Kp);
    uint8_t* out = P.x + size_t(u) * Geo::UNIT;
    const size_t from_step = size_t(stride) * (FPW * Kp), out_step = size_t(stride) * Geo::UNIT;
    if (u < units) load(from, frames_of(u));
    for (; u < units; u += stride, from += from_step, out += out_step) {
        const int count = frames_of(u), off = int(from & 15u);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < Geo::LOADS; ++k) {
            const int i = lane + 32 * k;
            const uint4 lo = raw[k][0], hi = raw[k][1];
            if (32 * i < off + count * Kp)
                bits[i] = pack4(lo.x) | (pack4(lo.y) << 4) | (pack4(lo.z) << 8) | (pack4(lo.w) << 12) | (pack4(hi.x) << 16) |
                          (pack4(hi.y) << 20) | (pack4(hi.z) << 24) | (pack4(hi.w) << 28);
        }
        __syncwarp();
        if (u + stride < units) load(from + from_step, frames_of(u + stride));
        const int fl = lane / LPF;                      // the lane's frame in the unit
        const int first = off + (fl < count ? fl : 0) * Kp;
        auto window = [&](int pos) { return __funnelshift_r(bits[pos >> 5], bits[(pos >> 5) + 1], unsigned(pos)); };
        // bits 0 .. n-1 of v, n in 0 .. 32
        auto low_bits = [](uint32_t v, int n) { return n >= 32 ? v : (n <= 0 ? 0u : v & ((1u << n) - 1u)); };
        uint32_t crc = 0;                               // remainder, bit j = its bit r-1-j
        if (r > 0) {
#pragma unroll
            for (int q = 0; q < WPL; ++q) {
                const int w = w0 + 32 * q;
                if (32 * w < Kp) {
                    const uint32_t v = low_bits(window(first + 32 * w), Kp - 32 * w);
#pragma unroll
                    for (int k = 0; k < 8; ++k) crc ^= table[(16 * k + int((v >> (4 * k)) & 15u)) * W + w];
                }
            }
            if constexpr (LPF == 32) {
                crc = __reduce_xor_sync(0xffffffffu, crc);
            } else {
#pragma unroll
                for (int o = LPF / 2; o > 0; o >>= 1) crc ^= __shfl_xor_sync(0xffffffffu, crc, o);
            }
            crc = __brev(crc) >> (32 - r);
        }
        uint32_t x[WPL];
#pragma unroll
        for (int q = 0; q < WPL; ++q) {
            // information bits rank .. of payload || CRC, moved to the word's information positions
            const int left = Kp - rank[q];              // payload bits from this rank on
            uint32_t v = low_bits(window(first + (left > 0 ? rank[q] : 0)), left);
            if (left < 32) v |= left >= 0 ? crc << left : (-left < 32 ? crc >> -left : 0u);
#pragma unroll
            for (int i = 4; i >= 0; --i) v = (v & ~step[q][i]) | ((v << (1 << i)) & step[q][i]);
            v &= info[q];
            // u G_N inside the word
            constexpr uint32_t clear[5] = {0x55555555u, 0x33333333u, 0x0F0F0F0Fu, 0x00FF00FFu, 0x0000FFFFu};
#pragma unroll
            for (int p = 0; p < (LOGN < 5 ? LOGN : 5); ++p) v ^= (v >> (1 << p)) & clear[p];
            x[q] = v;
        }
        // and between words
#pragma unroll
        for (int p = 5; p < LOGN && p < 10; ++p)
#pragma unroll
            for (int q = 0; q < WPL; ++q) {
                const uint32_t other = __shfl_xor_sync(0xffffffffu, x[q], 1 << (p - 5));
                if (!((w0 >> (p - 5)) & 1)) x[q] ^= other;
            }
        if constexpr (WPL == 2) x[0] ^= x[1];
        // codeword bytes
        const int bytes = count * N;
        if constexpr (N >= 32) {
#pragma unroll
            for (int q = 0; q < WPL; ++q)
                if constexpr (WIDE) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        // piece 32 h + lane of 16 bytes of the warp's 1 KB
                        const uint32_t v = __shfl_sync(0xffffffffu, x[q], 16 * h + (lane >> 1)) >> (16 * (lane & 1));
                        const int at = 1024 * q + 512 * h + 16 * lane;
                        if (at < bytes)
                            __stcs(reinterpret_cast<uint4*>(out + at),
                                   make_uint4(spread4(v), spread4(v >> 4), spread4(v >> 8), spread4(v >> 12)));
                    }
                } else {
                    // a word at a time, a byte a lane (98,309 frames of N = 1024, K = 512 off the boundary
                    // 65 us; with 16 bytes a lane one after another 306)
#pragma unroll 8
                    for (int i = 0; i < 32; ++i) {
                        const uint32_t v = __shfl_sync(0xffffffffu, x[q], i);
                        const int at = 1024 * q + 32 * i + lane;
                        if (at < bytes) out[at] = uint8_t((v >> lane) & 1u);
                    }
                }
        } else if (lane * N < bytes) {
            uint8_t* const o = out + lane * N;
            if constexpr (WIDE) {
#pragma unroll
                for (int b = 0; b < N; b += 8)
                    *reinterpret_cast<uint2*>(o + b) = make_uint2(spread4(x[0] >> b), spread4(x[0] >> (b + 4)));
            } else {
                for (int b = 0; b < N; ++b) o[b] = uint8_t((x[0] >> b) & 1u);
            }
        }
    }
}

constexpr int kEncodeCtas = 6;

template <int LOGN>
int launch_encode(const EncParams& P, int sms, cudaStream_t st)
{
    using Geo = EncGeo<LOGN>;
    static_assert(Geo::smem(Geo::N) <= 48 * 1024, "within the default limit of dynamic shared memory");
    const size_t smem = Geo::smem(P.K);
    // persistent CTAs (the table is made once per CTA; 4, 6 and 8 per SM measured alike)
    const int64_t tiles = (P.B + Geo::WARPS * Geo::FPW - 1) / (Geo::WARPS * Geo::FPW);
    const int grid = int(std::min<int64_t>(tiles, int64_t(sms) * kEncodeCtas));
    if ((reinterpret_cast<uintptr_t>(P.x) & 15u) == 0) encode_kernel<LOGN, true><<<grid, 256, smem, st>>>(P);
    else encode_kernel<LOGN, false><<<grid, 256, smem, st>>>(P);
    return cudaGetLastError() == cudaSuccess ? PC_OK : PC_ECUDA;
}

}  // namespace

}  // namespace pcbp

using namespace pcbp;

extern "C" int pc_encode(const pc_code* code, const uint8_t* d_payload, uint8_t* d_x, int64_t B, void* stream)
{
    int rc = validate_code(code);
    if (rc != PC_OK) return rc;
    if (B < 0) return PC_EINVAL;
    if (B == 0) return PC_OK;
    if (!d_x || (!d_payload && code->K - code->crc_len > 0)) return PC_EINVAL;
    DeviceInfo di;
    rc = device_info(&di);
    if (rc != PC_OK) return rc;
    std::unique_ptr<EncParams> P(new EncParams);
    build_enc_params(code, P.get());
    P->payload = d_payload;
    P->x = d_x;
    P->B = B;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    switch (code->n) {
        case 3: return launch_encode<3>(*P, di.sms, st);
        case 4: return launch_encode<4>(*P, di.sms, st);
        case 5: return launch_encode<5>(*P, di.sms, st);
        case 6: return launch_encode<6>(*P, di.sms, st);
        case 7: return launch_encode<7>(*P, di.sms, st);
        case 8: return launch_encode<8>(*P, di.sms, st);
        case 9: return launch_encode<9>(*P, di.sms, st);
        case 10: return launch_encode<10>(*P, di.sms, st);
        default: return launch_encode<11>(*P, di.sms, st);
    }
}
