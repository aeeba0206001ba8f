// ct.cu -- constant-time ECB: the bitsliced cipher of bitslice.cuh on GB300.
//
// Each thread owns 8 blocks at a time: lane l of a warp takes blocks base +
// 32 j + l, j = 0..7, so every warp-wide 128-bit load or store still covers
// 512 contiguous bytes.  The thread transposes its 32 words into 32 bit planes
// (word 8 c + j, column c of block j, becomes bit 8 c + j of every plane), runs
// the rounds as logic operations on whole planes, transposes back and stores.
// No address depends on key or data.  Round keys reach the circuits as mask
// planes built on the host from the schedule (one mask byte per byte position
// and key step, see build_masks) and expanded into shared memory at the start
// of the kernel.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#include "aes_kernels.cuh"
#include "bitslice.cuh"
#include "capi_internal.h"
#include "registry.h"

namespace aesgb {

constexpr int kCtThreads = 512;  // largest CTA (94 registers: one per SM)
constexpr int kCtBlocks = 8;  // AES blocks per thread and pass: one word per (row, bit) plane

struct CtArgs {
    const uint4 *in;
    uint4 *out;
    unsigned long long nblocks;
    int nr;
    uint8_t masks[15][16];  // [key step][byte q = r + 4c]
};

// Key bytes of steps 0..Nr as the kernel takes them (bitslice.cuh adds step 0
// to the input and gives step i to the circuits of round i).  K_i is round
// key i of the encryption schedule w, as a state (byte q = r + 4c is row r,
// column c); a byte m wanted at an S-box output is passed as mu = OUT^-1 m
// (bsc::k_mu_enc / k_mu_dec), which the S-box's product chains add for free.
//   encryption  step 0: K_0.  Round i adds its key at the S-box outputs,
//               before ShiftRows and MixColumns, together with the S-box's
//               constant 63: m[q] = 63 + K'_i[r + 4((c - r) mod 4)], where
//               K'_i = InvMixColumns(K_i) for i < Nr and K_Nr itself (the
//               last round has no MixColumns); ShiftRows then carries byte
//               (r, (c - r) mod 4) to (r, c), and MixColumns(K'_i) = K_i.
//   decryption  (inverse cipher, FIPS-197 5.3): step 0 is K_Nr; round i adds
//               K_{Nr-i} right after InvSubBytes, m = K_{Nr-i}, and the column
//               circuit applies InvMixColumns to the sum.
struct MuTables {
    uint8_t of[2][256];  // OUT^-1 m of the encryption and of the decryption S-box circuit
};
constexpr MuTables make_mu_tables() {
    MuTables t{};
    for (int m = 0; m < 256; ++m) {
        t.of[0][m] = bs::apply_rows(bsc::k_mu_enc, static_cast<uint8_t>(m));
        t.of[1][m] = bs::apply_rows(bsc::k_mu_dec, static_cast<uint8_t>(m));
    }
    return t;
}
constexpr MuTables kMu = make_mu_tables();

// MixColumns / InvMixColumns of one key column on the host, from the round
// tables: te0[x] is the MixColumns column of S(x) in row 0 (eq (22)), td0[x]
// the InvMixColumns column of InvS(x); rows 1..3 are byte rotations.
uint32_t key_column(const uint32_t (&tab)[256], const uint8_t (&undo)[256], const uint8_t *k) {
    uint32_t v = 0;
    for (int r = 0; r < 4; ++r) {
        const uint32_t t = tab[undo[k[r]]];
        v ^= r == 0 ? t : (t << (8 * r)) | (t >> (32 - 8 * r));
    }
    return v;
}

void build_masks(int dir, const uint32_t *rk, int nr, uint8_t (*out)[16]) {
    uint8_t w[240];
    std::memcpy(w, rk, 16 * (nr + 1));
    // encryption needs InvMixColumns of keys 1..Nr-1; dw (decryption) holds
    // InvMixColumns(w_r) there, and MixColumns gives w back
    uint8_t mixed[240];
    for (int q = 16; q < 16 * nr; q += 4) {
        const uint32_t col = dir == 0 ? key_column(kAes.td0, kAes.sbox, w + q) : key_column(kAes.te0, kAes.isbox, w + q);
        std::memcpy(mixed + q, &col, 4);
    }
    std::memcpy(mixed, w, 16);
    std::memcpy(mixed + 16 * nr, w + 16 * nr, 16);
    std::memcpy(out[0], mixed + (dir == 0 ? 0 : 16 * nr), 16);
    for (int i = 1; i <= nr; ++i)
        for (int q = 0; q < 16; ++q) {
            const int r = q & 3, c = q >> 2;
            const uint8_t m = dir == 0 ? static_cast<uint8_t>(0x63 ^ mixed[16 * i + r + 4 * ((c - r + 4) & 3)])
                                       : mixed[16 * (nr - i) + q];
            out[i][q] = kMu.of[dir][m];
        }
}

// Mask bytes -> planes, in the state's layout: plane p = 8 r + b of step i / 32,
// byte c all ones where bit b of the mask byte (r, c) is set.
AESGB_HD void expand_mask(const uint8_t (*m)[16], int i, bs::RoundMasks *dst) {
    const int app = i >> 5, p = i & 31, r = p >> 3, b = p & 7;
#if defined(__CUDA_ARCH__)
    if (!AESGB_CHECK(app < 15)) return;
#endif
    uint32_t v = 0;
    for (int c = 0; c < 4; ++c) v |= ((m[app][r + 4 * c] >> b) & 1u) * (0xffu << (8 * c));
    dst[app].m[p] = v;
}

// Bound: the integer-logic (ALU) pipe, 64 lanes per clock per SM: 527 counted
// operations per block for AES-128 encryption (aes_ct_ops_per_block), 30 byte
// permutes for ShiftRows and about 10 more for addresses and bounds.  A unit of
// work is a warp's 256 blocks (4 KiB).  8 blocks and 32 planes per thread take
// 94 registers without spill, and keep the pipe 98.8 % busy; the form with 32
// blocks and 128 planes, one word per (column, row, bit), needs no permutes but
// 255 registers and a unit of 16 KiB, so a pass was four times as long and a
// 1 MiB buffer filled 8 SMs.  Units go round the CTAs first and then the warps of
// each, so that every SM, and every quarter of one, gets the same number within
// one.  Measured against that form (replayed graph): AES-128 encryption 64 KiB
// 20.0 -> 5.7 us, 1 MiB 36.0 -> 5.7, 16 MiB 38.2 -> 33.9, 256 MiB 536 -> 492, 1
// GiB 1,987 -> 1,956, 8 GiB 16,190 -> 15,575; AES-256 decryption 256 MiB 753 ->
// 711, 8 GiB 23,273 -> 22,601.  The permutes grow with the rounds, so between
// 0.75 and 2.5 GiB, where the other form's last pass costs little and its clock
// has not come down yet, it was ahead at AES-256 (encryption 1 GiB 2,619 / 2,659,
// 2 GiB 5,231 / 5,304, 4 GiB 10,648 / 10,596; decryption by 0.5 to 1 %) and at
// AES-192 encryption (1.5 GiB 3,413 / 3,453).  A second kernel that spills for
// 1.7 % at most, in that window, is not kept.
template <int DIR>
__global__ void __launch_bounds__(kCtThreads, 1) ct_kernel(const __grid_constant__ CtArgs a) {
    __shared__ bs::RoundMasks masks[15];
    for (int i = threadIdx.x; i < (a.nr + 1) * 32; i += blockDim.x) expand_mask(a.masks, i, masks);
    __syncthreads();
    griddep_release();
    griddep_wait();  // global memory only after this (see aes_kernels.cuh)
    const uint32_t lane = threadIdx.x & 31u;
    constexpr unsigned long long kUnit = 32ull * kCtBlocks;  // blocks of a warp's pass
    const unsigned long long wpc = blockDim.x >> 5;
    const unsigned long long step = static_cast<unsigned long long>(gridDim.x) * wpc * kUnit;
    const unsigned long long n = a.nblocks;
    // units go round the CTAs first, then the warps of each
    for (unsigned long long base = (static_cast<unsigned long long>(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * kUnit;
         base < n; base += step) {
        bs::Planes s;
#pragma unroll
        for (int j = 0; j < kCtBlocks; ++j) {
            const unsigned long long blk = base + 32ull * j + lane;
            const uint4 v = blk < n ? ld_block(a.in + blk) : make_uint4(0, 0, 0, 0);
            s.w[j] = v.x;
            s.w[8 + j] = v.y;
            s.w[16 + j] = v.z;
            s.w[24 + j] = v.w;
        }
        bs::transpose32(s.w);
        bs::cipher_planes<DIR>(s, masks, a.nr);
        bs::transpose32(s.w);
#pragma unroll
        for (int j = 0; j < kCtBlocks; ++j) {
            const unsigned long long blk = base + 32ull * j + lane;
            if (blk < n) st_block(a.out + blk, make_uint4(s.w[j], s.w[8 + j], s.w[16 + j], s.w[24 + j]));
        }
    }
}

AESGB_BOUNDS_READER(ct)

}  // namespace aesgb

using namespace aesgb;

extern "C" {

int aes_ecb_crypt_ct(int dir, const uint32_t *rk, int nrounds, const uint8_t *in, uint8_t *out, size_t nblocks,
                     void *stream) {
    if (dir != 0 && dir != 1) return AES_E_ARG;
    int st = check_nrounds(nrounds);
    if (st != AES_OK) return st;
    if (!rk) return AES_E_ARG;
    if (nblocks == 0) return AES_OK;
    st = check_buffers(in, out, nblocks);
    if (st != AES_OK) return st;
    CtArgs args;
    std::memset(&args, 0, sizeof args);
    args.in = reinterpret_cast<const uint4 *>(in);
    args.out = reinterpret_cast<uint4 *>(out);
    args.nblocks = nblocks;
    args.nr = nrounds;
    build_masks(dir, rk, nrounds, args.masks);
    int dev = 0;
    if (current_device(&dev) != AES_OK) return AES_E_CUDA;
    const void *fn = dir == 0 ? reinterpret_cast<const void *>(&ct_kernel<0>)
                              : reinterpret_cast<const void *>(&ct_kernel<1>);
    const int sms = sm_count(dev);
    if (sms < 0) return sms;
    // One CTA per SM, or one per unit when there are fewer.  One warp per SM
    // quarter keeps the ALU pipe 94 % busy (its circuits are independent), so a
    // buffer with few units per SM gets a small CTA, whose registers leave room
    // for the next launch's to start behind it (programmatic dependent launch).
    // Up to four units per SM every warp of the CTA has one: two CTAs that meet on
    // an SM then use different quarters, where CTAs of four warps with two at work
    // put both on the same ones (1 MiB in a stream of launches: 5.8 us, or 8.5 to
    // 9.4 whenever the launches fell into that pattern).  Large buffers get 16
    // warps, which run closely enough together to share the instruction cache:
    // 256 MiB, AES-128 encryption, took 492.7 us with 512 threads, 502.1 with 256,
    // 507.2 with five CTAs of 128.
    const unsigned long long units = (nblocks + 32 * kCtBlocks - 1) / (32 * kCtBlocks);
    const unsigned long long per_sm = (units + sms - 1) / sms;
    const int threads = per_sm > 8 ? kCtThreads : per_sm > 4 ? 256 : static_cast<int>(32 * per_sm);
    const int grid = static_cast<int>(units < static_cast<unsigned long long>(sms) ? units : sms);
    void *params[] = {&args};
    return launch_pdl(fn, grid, threads, 0, params, stream);
}

int aes_ct_ops_per_block(int dir, int nrounds, double *ops_per_block) {
    if ((dir != 0 && dir != 1) || !ops_per_block) return AES_E_ARG;
    const int st = check_nrounds(nrounds);
    if (st != AES_OK) return st;
    // per thread and 8-block group: 32 planes of step-0 key, the rounds, 2
    // transposes of 32 words (stages 16 and 8: one byte permute per word,
    // stages 4, 2 and 1: one bit-select per word)
    long long g = 32 + 2 * (2 * 32 + 3 * 32);
    if (dir == 0)
        g += 4LL * nrounds * bsc::k_sbox_enc.kGates + (nrounds - 1LL) * bsc::k_mix_columns.kGates;
    else
        g += 4LL * nrounds * bsc::k_sbox_core_dec.kGates + (nrounds - 1LL) * bsc::k_inv_mix_out.kGates +
             4LL * bsc::k_sbox_out_dec.kGates;
    *ops_per_block = static_cast<double>(g) / kCtBlocks;
    return AES_OK;
}

int aes_ct_selftest_host(int dir, const uint32_t *rk, int nrounds, const uint8_t *in, uint8_t *out,
                         size_t nblocks) {
    if ((dir != 0 && dir != 1) || !rk || (nblocks && (!in || !out))) return AES_E_ARG;
    int st = check_nrounds(nrounds);
    if (st != AES_OK) return st;
    uint8_t mb[15][16];
    build_masks(dir, rk, nrounds, mb);
    bs::RoundMasks masks[15];
    for (int i = 0; i < (nrounds + 1) * 32; ++i) expand_mask(mb, i, masks);
    for (size_t g = 0; g < nblocks; g += kCtBlocks) {
        bs::Planes s;
        for (int j = 0; j < kCtBlocks; ++j) {
            uint32_t v[4] = {0, 0, 0, 0};
            if (g + j < nblocks) std::memcpy(v, in + 16 * (g + j), 16);
            for (int c = 0; c < 4; ++c) s.w[8 * c + j] = v[c];
        }
        bs::transpose32(s.w);
        if (dir == 0) bs::cipher_planes<0>(s, masks, nrounds);
        else bs::cipher_planes<1>(s, masks, nrounds);
        bs::transpose32(s.w);
        for (int j = 0; j < kCtBlocks; ++j) {
            if (g + j >= nblocks) break;
            uint32_t v[4];
            for (int c = 0; c < 4; ++c) v[c] = s.w[8 * c + j];
            std::memcpy(out + 16 * (g + j), v, 16);
        }
    }
    return AES_OK;
}

}  // extern "C"
