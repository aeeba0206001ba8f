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
    uint32_t passes;                    // passes of 32 * NB blocks per unit: 1, 2, 4 or 8, at most 256 blocks
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
#define AESGB_M(KERNEL, NR, L) \
    if (nr == NR && layout == L) return reinterpret_cast<const void *>(&KERNEL<NR, 1, L>);
#define AESGB_C(MODE, NR, L) \
    if (nr == NR && layout == L) return reinterpret_cast<const void *>(&chain_dec_kernel<MODE, NR, 1, L>);

const void *ctr_kernel_ptr(int nr, int layout) {
    AESGB_M(ctr_kernel, 10, kLayoutR4) AESGB_M(ctr_kernel, 12, kLayoutR4) AESGB_M(ctr_kernel, 14, kLayoutR4)
    AESGB_M(ctr_kernel, 10, kLayoutR2) AESGB_M(ctr_kernel, 12, kLayoutR2) AESGB_M(ctr_kernel, 14, kLayoutR2)
    return nullptr;
}

const void *cbc_dec_kernel_ptr(int nr, int layout) {
    AESGB_C(kChainCbc, 10, kLayoutR2) AESGB_C(kChainCbc, 12, kLayoutR2) AESGB_C(kChainCbc, 14, kLayoutR2)
    AESGB_C(kChainCbc, 10, kLayoutR4) AESGB_C(kChainCbc, 12, kLayoutR4) AESGB_C(kChainCbc, 14, kLayoutR4)
    return nullptr;
}

const void *cfb_dec_kernel_ptr(int nr, int layout) {
    AESGB_C(kChainCfb, 10, kLayoutR4) AESGB_C(kChainCfb, 12, kLayoutR4) AESGB_C(kChainCfb, 14, kLayoutR4)
    AESGB_C(kChainCfb, 10, kLayoutR2) AESGB_C(kChainCfb, 12, kLayoutR2) AESGB_C(kChainCfb, 14, kLayoutR2)
    return nullptr;
}

namespace {

// Launch shape of a mode: one CTA of 1,024 threads per SM with R4 tables from
// 1,024 blocks per SM up; below that R2, 512 threads, as many CTAs as fit.
// Before, one CTA of 256 threads with R4 tables ran up to 16,384 blocks per SM
// (40 MiB): 8 warps, too few to keep the data pipe full.  Replayed graph,
// AES-128, 16 MiB: CBC 27.4 -> 21.9 us, CFB 26.2 -> 21.5; 4 MiB: CBC 8.9 -> 8.0,
// CFB 8.6 -> 7.5.  R2 instead of R4: 197 MiB CBC 235.0 / 234.4 us, CFB 235.5 /
// 232.7.  The line itself: 512 against 1,024 threads CBC 4.61 / 4.71 us at 2 MiB,
// 7.30 / 7.16 at 4 MiB.
aes_launch_cfg mode_cfg(size_t nblocks) {
    int dev = 0;
    const int sms = current_device(&dev) == AES_OK ? sm_count(dev) : 0;
    const bool large = nblocks >= static_cast<size_t>(sms > 0 ? sms : 152) * 1024;
    aes_launch_cfg c;
    c.layout = large ? AES_LAYOUT_R4 : AES_LAYOUT_R2;
    c.threads = large ? 1024 : 512;
    c.blocks_per_thread = 1;
    c.ctas_per_sm = 0;
    return c;
}

// Passes of a CTR unit: as many as give every warp one unit, up to the 8 of a
// whole 256-block group; above that 4 until the units are many, so that the
// last round of units is short.  AES-128, 1,024 threads (1 / 2 / 4 / 8 passes):
// 4 MiB 6.9 / 6.75 / 6.9 / - us, 8 MiB 11.1 / 10.96 / 10.54 / -, 16 MiB 18.9 /
// 18.6 / 18.6 / 18.4, 32 MiB - / 34.1 / 34.0 / 34.3, 256 MiB - / 253.1 / 249.9 /
// 248.6.
uint32_t ctr_passes(const aes_launch_cfg &c, int grid, size_t nblocks) {
    const unsigned long long per_pass = static_cast<unsigned long long>(grid) * static_cast<unsigned int>(c.threads);
    const unsigned long long r = (nblocks + per_pass - 1) / per_pass;  // passes if every warp takes the same
    return r > 32 ? 8u : r > 8 ? 4u : r > 4 ? 8u : r > 2 ? 4u : r > 1 ? 2u : 1u;
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
    const aes_launch_cfg c = mode_cfg(nblocks);
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
    return launch_mode(ctr_kernel_ptr(nrounds, c.layout), kEncrypt, c, nblocks, args, stream,
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
    const aes_launch_cfg c = mode_cfg(nblocks);
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
    const aes_launch_cfg c = mode_cfg(nblocks);
    CbcArgs args;
    args.in = reinterpret_cast<const uint4 *>(in);
    args.out = reinterpret_cast<uint4 *>(out);
    args.nblocks = nblocks;
    order_round_keys(kEncrypt, rk_enc, nrounds, &args.rk);
    std::memcpy(&args.iv, iv, 16);
    return launch_mode(cfb_dec_kernel_ptr(nrounds, c.layout), kEncrypt, c, nblocks, args, stream, [](int) {});
}

}  // extern "C"
