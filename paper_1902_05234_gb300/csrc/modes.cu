// modes.cu -- the other block-parallel uses of the T-table cipher:
//
//  CTR (Wang & Chu section 3.1.5, eq (5); Table 1 marks it, with ECB, as
//  suitable for parallel execution): C_i = P_i xor E(counter block of block i),
//  the counter block of block i being the caller's first counter block plus i
//  as a 128-bit big-endian integer (mod 2^128).  Encryption and decryption are
//  the same operation.
//
//  CBC decryption (section 3.1.2; eq (2) as printed omits the cipher, the
//  reading is P_i = D(C_i) xor C_{i-1}, C_{-1} = IV).  Encryption chains and
//  stays sequential (Table 1), but every decryption step needs only two
//  ciphertext blocks, so it parallelises like ECB: lane l of a warp takes the
//  previous ciphertext block from lane l-1 by a shuffle, lane 0 from lane 31
//  of the previous slice or from memory / the IV.
//
// Both reuse the bank-replicated tables and the round code of ECB; round keys
// and the counter / IV travel in the kernel parameters (constant bank).
#include <cstring>

#include "aes_kernels.cuh"
#include "capi_internal.h"
#include "registry.h"

namespace aesgb {

struct CtrArgs {
    const uint4 *in;
    uint4 *out;
    unsigned long long nblocks;
    RoundKeys rk;
    unsigned long long ctr_hi, ctr_lo;  // first counter block as a 128-bit integer
    uint32_t passes;                    // passes of 32 * NB blocks per unit: 2, 4 or 8, at most 256 blocks
};

struct CbcArgs {
    const uint4 *in;
    uint4 *out;
    unsigned long long nblocks;
    RoundKeys rk;
    uint4 iv;
};

__device__ __forceinline__ uint32_t bswap32(uint32_t v) { return __byte_perm(v, 0u, 0x0123u); }

// Counter block ctr + i as four state words (byte 0 of the block = most
// significant byte of the integer).
__device__ __forceinline__ void counter_state(unsigned long long hi, unsigned long long lo, unsigned long long i,
                                              uint32_t (&s)[4]) {
    const unsigned long long l = lo + i;
    const unsigned long long h = hi + (l < lo ? 1ull : 0ull);
    s[0] = bswap32(static_cast<uint32_t>(h >> 32));
    s[1] = bswap32(static_cast<uint32_t>(h));
    s[2] = bswap32(static_cast<uint32_t>(l >> 32));
    s[3] = bswap32(static_cast<uint32_t>(l));
}

// What 256 consecutive counter blocks with the same upper 15 bytes share.  The
// last byte sits in row 3, column 3; after ShiftRows it enters column 0 of round
// 1 only, and that column enters each column of round 2 in one row.  So
// columns 1..3 of round 1 and three of the four lookups of every column of
// round 2 are the same for all 256 blocks:
//   round 1  column 0 = r1 ^ T3[last byte ^ key byte], columns 1..3 fixed
//   round 2  column j = r2[j] ^ T_r[row r of round 1's column 0], r = -j mod 4.
// A block then costs 5 lookups for rounds 1 and 2 instead of 32.
struct CtrShared {
    uint32_t r1, r2[4];
};

template <int LAYOUT, class Key>
__device__ __forceinline__ CtrShared ctr_shared(const Tab<LAYOUT, kEncrypt> &tab, const Key &k, unsigned long long hi,
                                                unsigned long long lo, unsigned long long first) {
    uint32_t s[4], c[4];
    counter_state(hi, lo, first, s);
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] ^= k(j);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        c[j] = k(4 + j);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (j != 0 || r != 3) c[j] ^= lookup_t(tab, r, s[src_col<kEncrypt>(j, r)], r);
    }
    CtrShared v;
    v.r1 = c[0];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        v.r2[j] = k(8 + j);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (src_col<kEncrypt>(j, r) != 0) v.r2[j] ^= lookup_t(tab, r, c[src_col<kEncrypt>(j, r)], r);
    }
    return v;
}

// Bound: the L1TEX data pipe, 133 lookups per block at AES-128 instead of 160
// (197 instead of 224 at AES-256), plus 27/32 + 5 for each unit and the 8
// wavefronts of 32 blocks' input and output.  256 MiB, replayed graph: AES-128
// 289.7 -> 248.6 us (8,639 Gbit/s), AES-256 394.1 -> 352.0.
//
// A warp's unit is 32 * NB * a.passes consecutive counter blocks, a power of two
// of at most 256 and aligned to its size in the counter's last byte, so a unit
// shares the upper 15 bytes; the buffer's first and last unit may be partial.
// Lane i computes what the unit i units ahead shares, for 32 units at once, and
// the warp takes it from there by shuffles.
template <int NR, int NB, int LAYOUT>
__global__ void __launch_bounds__(max_threads_for_nb(NB), 1) ctr_kernel(const __grid_constant__ CtrArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned long long W = static_cast<unsigned long long>(gridDim.x) * (blockDim.x >> 5);
    const uint32_t unit = 32u * NB * a.passes;
    // blocks are numbered from the start of the first one's 256-block group
    const uint32_t skip = static_cast<uint32_t>(a.ctr_lo) & 255u;
    const unsigned long long lo = a.ctr_lo - skip, end = a.nblocks + skip;
    const unsigned long long U = (end + unit - 1) / unit;
    unsigned long long u = static_cast<unsigned long long>(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    Tab<LAYOUT, kEncrypt>::fill(smem, threadIdx.x, blockDim.x);
    __syncthreads();
    griddep_release();
    griddep_wait();  // global memory only after this (see aes_kernels.cuh)
    auto load = [&](unsigned long long v, uint4 (&x)[NB]) {
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const unsigned long long b = v + 32ull * i;
            x[i] = b >= skip && b < end ? ld_block(a.in + (b - skip)) : make_uint4(0, 0, 0, 0);
        }
    };
    uint4 cur[NB];
    load(u * unit + lane, cur);
    const Tab<LAYOUT, kEncrypt> tab(smem, lane);
    const ParamKey key{a.rk.w};
    while (u < U) {
        const CtrShared mine = ctr_shared(tab, key, a.ctr_hi, lo, ((u + lane * W) * unit) & ~255ull);
        for (int i = 0; i < 32 && u < U; ++i, u += W) {
            CtrShared sh;
            sh.r1 = __shfl_sync(0xffffffffu, mine.r1, i);
#pragma unroll
            for (int j = 0; j < 4; ++j) sh.r2[j] = __shfl_sync(0xffffffffu, mine.r2[j], i);
            unsigned long long v = u * unit + lane;
            for (uint32_t p = 0; p < a.passes; ++p) {
                const unsigned long long next = p + 1 < a.passes ? v + 32u * NB : (u + W) * unit + lane;
                uint4 nxt[NB];
                load(next, nxt);
                uint32_t s[NB][4];
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    const uint32_t last = (static_cast<uint32_t>(v + 32u * q) << 24) ^ key(3);  // byte 3 is used
                    const uint32_t c0 = sh.r1 ^ lookup_t(tab, 3, last, 3);
#pragma unroll
                    for (int j = 0; j < 4; ++j) s[q][j] = sh.r2[j] ^ lookup_t(tab, (4 - j) & 3, c0, (4 - j) & 3);
                }
                cipher_rounds<kEncrypt, NR, NB, 3>(tab, key, s);
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    const unsigned long long b = v + 32ull * q;
                    if (b >= skip && b < end)
                        st_block(a.out + (b - skip), make_uint4(cur[q].x ^ s[q][0], cur[q].y ^ s[q][1],
                                                                cur[q].z ^ s[q][2], cur[q].w ^ s[q][3]));
                    cur[q] = nxt[q];
                }
                v = next;
            }
        }
    }
}

// Up to a block per thread and 1,024 per SM: no shared rounds.  What 256 blocks
// share would be computed for a unit of 32, ahead of the unit's own rounds, and
// the time of such a call is one warp's chain of rounds.  A stream of launches
// (replayed graph), this kernel against the shared form with 512 threads and R2
// tables: 64 KiB AES-128 3.43 -> 1.78 us, AES-256 4.18 -> 2.07; 1 MiB 4.56 ->
// 2.79 and 5.67 -> 3.28; 2 MiB 4.62 -> 3.98.  At 2.5 MiB the shared form takes
// over (4.95 against 5.04 us).
template <int NR, int LAYOUT>
__global__ void __launch_bounds__(max_threads_for_nb(1), 1) ctr_small_kernel(const __grid_constant__ CtrArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned long long step = static_cast<unsigned long long>(gridDim.x) * blockDim.x;
    Tab<LAYOUT, kEncrypt>::fill(smem, threadIdx.x, blockDim.x);
    __syncthreads();
    griddep_release();
    griddep_wait();  // global memory only after this (see aes_kernels.cuh)
    const Tab<LAYOUT, kEncrypt> tab(smem, lane);
    const ParamKey key{a.rk.w};
    for (unsigned long long b = static_cast<unsigned long long>(blockIdx.x) * blockDim.x + threadIdx.x; b < a.nblocks;
         b += step) {
        const uint4 v = ld_block(a.in + b);
        uint32_t s[1][4];
        counter_state(a.ctr_hi, a.ctr_lo, b, s[0]);
        cipher_states<kEncrypt, NR, 1>(tab, key, s);
        st_block(a.out + b, make_uint4(v.x ^ s[0][0], v.y ^ s[0][1], v.z ^ s[0][2], v.w ^ s[0][3]));
    }
}

__device__ __forceinline__ uint4 shfl_up1(uint4 v) {
    return make_uint4(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1),
                      __shfl_up_sync(0xffffffffu, v.z, 1), __shfl_up_sync(0xffffffffu, v.w, 1));
}
__device__ __forceinline__ uint4 shfl_from31(uint4 v) {
    return make_uint4(__shfl_sync(0xffffffffu, v.x, 31), __shfl_sync(0xffffffffu, v.y, 31),
                      __shfl_sync(0xffffffffu, v.z, 31), __shfl_sync(0xffffffffu, v.w, 31));
}

// Decryption of the two chained modes whose decryption is parallel (section
// 3.1.2-3.1.3, Table 1 marks their encryption unsuitable): each plaintext
// block needs its ciphertext block C_i and the one before, C_{i-1} (the IV
// before block 0).
//   CBC  P_i = D(C_i) xor C_{i-1}   (inverse cipher on the current block)
//   CFB  P_i = C_i xor E(C_{i-1})   (forward cipher on the previous block)
enum : int { kChainCbc = 0, kChainCfb = 1 };

template <int MODE, int NR, int NB, int LAYOUT>
__global__ void __launch_bounds__(max_threads_for_nb(NB), 1) chain_dec_kernel(const __grid_constant__ CbcArgs a) {
    constexpr int DIR = MODE == kChainCbc ? kDecrypt : kEncrypt;
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned long long n = a.nblocks;
    const unsigned long long step = static_cast<unsigned long long>(gridDim.x) * (blockDim.x >> 5) * 32ull * NB;
    // Slices go round the CTAs first, as in ecb_kernel, while they make at most
    // eight rounds of the grid; with more, CTA by CTA: the block before a slice is
    // then in another warp's lines of the same SM (197 MiB, R4: CBC 236.9 -> 234.4
    // us at AES-128, 319.1 -> 316.5 at AES-256).
    const unsigned long long wpc = blockDim.x >> 5, warp = threadIdx.x >> 5;
    unsigned long long base = (n <= 8 * step ? warp * gridDim.x + blockIdx.x : blockIdx.x * wpc + warp) * 32ull * NB;
    Tab<LAYOUT, DIR>::fill(smem, threadIdx.x, blockDim.x);
    __syncthreads();
    griddep_release();
    griddep_wait();  // global memory only after this (see aes_kernels.cuh)
    // the ciphertext block just before a slice (lane 0's chaining value; the
    // IV before block 0), loaded one pass ahead like the slice itself
    auto before = [&](unsigned long long b) {
        return b == 0 ? a.iv
                      : (lane == 0 && b < n && AESGB_CHECK(b - 1 < n) ? ld_block(a.in + (b - 1))
                                                                       : make_uint4(0, 0, 0, 0));
    };
    uint4 cur[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        const unsigned long long b = base + lane + 32ull * i;
        cur[i] = b < n ? ld_block(a.in + b) : make_uint4(0, 0, 0, 0);
    }
    uint4 before_cur = before(base);
    const Tab<LAYOUT, DIR> tab(smem, lane);
    const ParamKey key{a.rk.w};
    for (; base < n; base += step) {
        uint4 nxt[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const unsigned long long b = base + step + lane + 32ull * i;
            nxt[i] = b < n ? ld_block(a.in + b) : make_uint4(0, 0, 0, 0);
        }
        const uint4 before_nxt = before(base + step);
        // chaining values: the ciphertext block just before each of ours
        uint4 prev[NB];
        const uint4 before_slice0 = before_cur;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const uint4 up = shfl_up1(cur[i]);
            const uint4 from_prev_slice = i == 0 ? before_slice0 : shfl_from31(cur[i > 0 ? i - 1 : 0]);
            prev[i] = lane == 0 ? from_prev_slice : up;
        }
        uint32_t s[NB][4];
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const uint4 x = MODE == kChainCbc ? cur[i] : prev[i];  // the block the cipher runs on
            s[i][0] = x.x; s[i][1] = x.y; s[i][2] = x.z; s[i][3] = x.w;
        }
        cipher_states<DIR, NR, NB>(tab, key, s);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const unsigned long long b = base + lane + 32ull * i;
            const uint4 y = MODE == kChainCbc ? prev[i] : cur[i];  // the block XORed onto its output
            if (b < n) st_block(a.out + b, make_uint4(y.x ^ s[i][0], y.y ^ s[i][1], y.z ^ s[i][2], y.w ^ s[i][3]));
            cur[i] = nxt[i];
        }
        before_cur = before_nxt;
    }
}

AESGB_BOUNDS_READER(modes)

// One block per thread: two at 1,024 threads measured 0.2 % (CFB) to 2 % (CBC)
// slower at 256 MiB, AES-128, two at 512 threads 1-4 %.
#define AESGB_M(KERNEL, ...) return reinterpret_cast<const void *>(&KERNEL<__VA_ARGS__>)
#define AESGB_C(MODE, NR, L) \
    if (nr == NR && layout == L) return reinterpret_cast<const void *>(&chain_dec_kernel<MODE, NR, 1, L>);

const void *ctr_kernel_ptr(int nr, bool shared) {
    switch (nr) {
    case 10: if (shared) AESGB_M(ctr_kernel, 10, 1, kLayoutR4); else AESGB_M(ctr_small_kernel, 10, kLayoutR4);
    case 12: if (shared) AESGB_M(ctr_kernel, 12, 1, kLayoutR4); else AESGB_M(ctr_small_kernel, 12, kLayoutR4);
    case 14: if (shared) AESGB_M(ctr_kernel, 14, 1, kLayoutR4); else AESGB_M(ctr_small_kernel, 14, kLayoutR4);
    default: return nullptr;
    }
}

const void *cbc_dec_kernel_ptr(int nr, int layout) {
    AESGB_C(kChainCbc, 10, kLayoutR2) AESGB_C(kChainCbc, 12, kLayoutR2) AESGB_C(kChainCbc, 14, kLayoutR2)
    AESGB_C(kChainCbc, 10, kLayoutR4) AESGB_C(kChainCbc, 12, kLayoutR4) AESGB_C(kChainCbc, 14, kLayoutR4)
    return nullptr;
}

const void *cfb_dec_kernel_ptr(int nr, int layout) {
    AESGB_C(kChainCfb, 10, kLayoutR4) AESGB_C(kChainCfb, 12, kLayoutR4) AESGB_C(kChainCfb, 14, kLayoutR4)
    return nullptr;
}

namespace {

size_t blocks_per_sm(size_t nblocks) {  // rounded up
    int dev = 0;
    const int found = current_device(&dev) == AES_OK ? sm_count(dev) : 0;
    const size_t sms = static_cast<size_t>(found > 0 ? found : 152);
    return nblocks / sms + (nblocks % sms != 0);
}

// Launch shape of a mode, by blocks per SM.  One CTA per SM with R4
// tables and one block per thread, of as many warps as an SM's share has: 256
// threads up to 256 blocks per SM, 1,024 from 1,024 up.  R4 tables keep a second
// CTA off the SM, so a small call spreads over as many SMs as it has CTAs; with
// R2 tables and 512 threads it sat on half as many, up to three CTAs to an SM,
// and a launch of the stream could meet the one before it there.  Replayed
// graph, AES-128, 512 threads with R2 -> this: CFB 64 KiB 2.72 -> 1.78 us, 1 MiB
// 3.2 to 4.5 -> 2.88, 2 MiB 6.0 -> 4.15; CBC 64 KiB 2.74 -> 2.02, 0.5 MiB 2.75
// -> 2.45.  One CTA of 256 threads at all sizes: CFB 16 MiB 26.2 us against 21.5.
//
// CBC between 256 and 1,024 blocks per SM: its decryption tables take 160 KiB in
// R4, whose fill shows there.  R2, and 512 threads from 384 blocks per SM:
// 0.75 MiB (352 threads) 2.63 us with R2, 2.80 with R4, 2.78 with 512 threads
// and R2; 1 MiB 3.05 / 3.24 / 2.91.
aes_launch_cfg mode_cfg(bool cbc, size_t per_sm) {
    const size_t share = per_sm < 256 ? 256 : per_sm > 1024 ? 1024 : (per_sm + 31) / 32 * 32;
    const bool r2 = cbc && per_sm > 256 && per_sm <= 1024;
    aes_launch_cfg c;
    c.layout = r2 ? AES_LAYOUT_R2 : AES_LAYOUT_R4;
    c.threads = static_cast<int32_t>(r2 && per_sm > 384 ? 512 : share);
    c.blocks_per_thread = 1;
    c.ctas_per_sm = 0;
    return c;
}

// Passes of a CTR unit: as many as give every warp one unit, up to the 8 of a
// whole 256-block group; above that 4 until the units are many, so that the
// last round of units is short.  AES-128, 1,024 threads (1 / 2 / 4 / 8 passes):
// 4 MiB 6.9 / 6.75 / 6.9 / - us, 8 MiB 11.1 / 10.96 / 10.54 / -, 16 MiB 18.9 /
// 18.6 / 18.6 / 18.4, 32 MiB - / 34.1 / 34.0 / 34.3, 256 MiB - / 253.1 / 249.9 /
// 248.6.  (More than 1,024 blocks per SM: two passes at least.)
uint32_t ctr_passes(const aes_launch_cfg &c, int grid, size_t nblocks) {
    const unsigned long long per_pass = static_cast<unsigned long long>(grid) * static_cast<unsigned int>(c.threads);
    const unsigned long long r = (nblocks + per_pass - 1) / per_pass;  // passes if every warp takes the same
    return r > 32 ? 8u : r > 8 ? 4u : r > 4 ? 8u : r > 2 ? 4u : 2u;
}

// Grid and launch of a mode kernel; `set` is called with the grid first.
template <class Args, class Set>
int launch_mode(const void *fn, int dir, const aes_launch_cfg &c, size_t nblocks, Args &args, void *stream, Set set) {
    if (!fn) return AES_E_CONFIG;
    int dev = 0;
    if (current_device(&dev) != AES_OK) return AES_E_CUDA;
    const uint32_t smem = table_smem_bytes(dir, c.layout);
    int grid = 0;
    int st = persistent_grid(fn, dev, c, smem, static_cast<unsigned long long>(c.threads), nblocks, &grid);
    if (st != AES_OK) return st;
    set(grid);
    void *params[] = {&args};
    return launch_pdl(fn, grid, c.threads, smem, params, stream);
}

}  // namespace
}  // namespace aesgb

using namespace aesgb;

extern "C" {

int aes_ctr_crypt(const uint32_t *rk, int nrounds, const uint8_t *ctr0, const uint8_t *in, uint8_t *out,
                  size_t nblocks, void *stream) {
    int st = check_nrounds(nrounds);
    if (st != AES_OK) return st;
    if (!rk || !ctr0) return AES_E_ARG;
    if (nblocks == 0) return AES_OK;
    st = check_buffers(in, out, nblocks);
    if (st != AES_OK) return st;
    const size_t per_sm = blocks_per_sm(nblocks);
    const aes_launch_cfg c = mode_cfg(false, per_sm);
    CtrArgs args;
    args.in = reinterpret_cast<const uint4 *>(in);
    args.out = reinterpret_cast<uint4 *>(out);
    args.nblocks = nblocks;
    order_round_keys(kEncrypt, rk, nrounds, &args.rk);
    unsigned long long hi = 0, lo = 0;
    for (int b = 0; b < 8; ++b) hi = (hi << 8) | ctr0[b];
    for (int b = 8; b < 16; ++b) lo = (lo << 8) | ctr0[b];
    args.ctr_hi = hi;
    args.ctr_lo = lo;
    return launch_mode(ctr_kernel_ptr(nrounds, per_sm > 1024), kEncrypt, c, nblocks, args, stream,
                       [&](int grid) { args.passes = ctr_passes(c, grid, nblocks); });
}

int aes_cbc_decrypt(const uint32_t *rk_dec, int nrounds, const uint8_t *iv, const uint8_t *in, uint8_t *out,
                    size_t nblocks, void *stream) {
    int st = check_nrounds(nrounds);
    if (st != AES_OK) return st;
    if (!rk_dec || !iv) return AES_E_ARG;
    if (nblocks == 0) return AES_OK;
    st = check_buffers(in, out, nblocks);
    if (st != AES_OK) return st;
    if (in == out) return AES_E_OVERLAP;  // a block's ciphertext is still needed after its plaintext is written
    const aes_launch_cfg c = mode_cfg(true, blocks_per_sm(nblocks));
    CbcArgs args;
    args.in = reinterpret_cast<const uint4 *>(in);
    args.out = reinterpret_cast<uint4 *>(out);
    args.nblocks = nblocks;
    order_round_keys(kDecrypt, rk_dec, nrounds, &args.rk);
    std::memcpy(&args.iv, iv, 16);
    return launch_mode(cbc_dec_kernel_ptr(nrounds, c.layout), kDecrypt, c, nblocks, args, stream, [](int) {});
}

int aes_cfb_decrypt(const uint32_t *rk_enc, int nrounds, const uint8_t *iv, const uint8_t *in, uint8_t *out,
                    size_t nblocks, void *stream) {
    int st = check_nrounds(nrounds);
    if (st != AES_OK) return st;
    if (!rk_enc || !iv) return AES_E_ARG;
    if (nblocks == 0) return AES_OK;
    st = check_buffers(in, out, nblocks);
    if (st != AES_OK) return st;
    if (in == out) return AES_E_OVERLAP;  // as CBC: C_i is read again after P_i would overwrite it
    const aes_launch_cfg c = mode_cfg(false, blocks_per_sm(nblocks));
    CbcArgs args;
    args.in = reinterpret_cast<const uint4 *>(in);
    args.out = reinterpret_cast<uint4 *>(out);
    args.nblocks = nblocks;
    order_round_keys(kEncrypt, rk_enc, nrounds, &args.rk);
    std::memcpy(&args.iv, iv, 16);
    return launch_mode(cfb_dec_kernel_ptr(nrounds, c.layout), kEncrypt, c, nblocks, args, stream, [](int) {});
}

}  // extern "C"
