// Prompt-end pass, bf16, many recorded rows (wide windows, groups): phases A and B of corm_prompt.cuh on tcgen05.
//
// A unit's rows go through 128 at a time: a row is a lane of tensor memory, a key of the tile (64 keys) a column, so a thread
// owns one row: its sum of exponentials is one fp64 register, its threshold and bounds are constants, and no sum crosses lanes.
// Operands lie in shared memory with the 128-byte swizzle: the rows' pieces q1, q2, q3 (96 KB at 128 channels) and, two tiles
// deep, the keys' pieces k1, k2, r2 (48 KB each), cut once per 128 rows (mma.sync: per 16) by the threads that load the keys,
// eight keys of a warp on one grid. Phase A accumulates the seven products of pieces (corm_mma.cuh) in four accumulators of
// 64 columns, two tiles of them in the 512 columns of tensor memory, so that one tile's products are issued (by a ninth warp)
// while the block's eight warps cut the next and take the exponentials of the one before. Phase B: one product of the raw
// values, verdicts by ballot; the logits inside the rounding bound are listed and formed again in fp64, four lanes each.
//
// Accumulation on tcgen05, checked on the GPU as for mma.sync (tests/test_gpu_tc_products.py for what the pieces reach): whole
// numbers up to 2^23.8, chains of 56, random and of one sign, none off by a bit. Accumulators: k1.q1; k1.q2 + k2.q1; k2.q2 (all exact); k1.q3, then r2.q2, then r2.q1. The last one is
// rounded: with 17 roundings of 2^-23 a step on what has been added up so far, its eight steps of r2.q1 err by at most
// 8 x 17 x 2^-23 A |q1|_1 / 8192, the smaller terms before them by 24 and 16 times 17 x 2^-23 of theirs (tc_split_error).
//
// What bounds it: fp64 and tensor instructions share a pipe, so phase A takes the products' time plus the exponentials'.
// 512 rows x 1024 keys a block, us: phase A 302 (163 with the exponentials left out, 173 with the products left out, 75 with
// both), phase B 121. Hence few fp64 operations per row and key: 13 with a table of 2^(i/16) and the 1/sqrt(d) inside the constants, 20
// before; and few integer ones, which issue as slowly (masks only on the last keys, ballots through shared memory: phase B 173
// -> 121). us per pass, mma.sync -> here: 128 units x 2048..4096 keys, G 1, w 256, 1580 -> 905; 32 units x 8192 keys, G 4, w
// 128, 1657 -> 1045; 8 units x 4096, w 128, 160 -> 89. Tried: the products issued by one of the eight warps in turn (the same).
#pragma once

#include <type_traits>

#include "corm_prompt_rows.cuh"

namespace corm {

constexpr int kTcRows = 128, kTcKeys = 64;
constexpr int kTcMaxRows = 1024;                 // rows of a unit whose sums and thresholds fit next to the operands
constexpr int kTcNearFlush = 2048, kTcNearCap = kTcNearFlush + kTcRows * kTcKeys;      // listed logits: a tile's always fit
constexpr int kTcThreads = kPcThreads + 32;      // a ninth warp issues phase A's products
constexpr int kTcStagesB = 4;
constexpr int kTcRowRoom = 4;                    // units of four rows that a warp of pc_fp64_rows keeps widened (little L1 is left)
// A block takes all of an SM's tensor memory and keeps it while it meets its cluster. A second one on the SM would wait for
// columns that the first gives back only after meeting peers that may wait in the same way, without end: so a block asks for
// more than half of the SM's shared memory (228 KB, of which the system takes 1 KB per block), whatever its operands need.
constexpr int kTcMinSmem = 114 * 1024;
static_assert(2 * (kTcMinSmem + 1024) > 228 * 1024, "two blocks must not fit an SM");

template <int D> struct TcShape {
    static constexpr int kSteps = D / 16, kBlocks = D / 64;               // 16-channel steps, 128-byte wide blocks of an operand
    static constexpr int kRowBlock = kTcRows * 128, kKeyBlock = kTcKeys * 128;
    static constexpr int kRowPiece = kBlocks * kRowBlock, kKeyPiece = kBlocks * kKeyBlock, kStage = 3 * kKeyPiece;
    static constexpr int kOperands = 3 * kRowPiece + 2 * kStage;
    static constexpr int kLoads = D / 32;        // 16-byte pieces of a tile per thread
};

struct TcMisc {
    unsigned long long bar[2], full[2];          // a tile's products are done; its pieces are there (and its accumulators free)
    double z[2][2][kTcRows];                     // phase A: a row's sums over the two halves of the tiles; by turns
    double exp16[16];                            // 2^(i / 16), i << 16 taken from the high words (TcExp)
    float scale[kTcStagesB][8];                  // per tile: largest magnitudes of its groups of eight keys (phase B)
    uint32_t words[2][kTcKeys];                  // phase B: the tiles' registers
    uint32_t who[kPcWarps][32];                  // rows of the warp that find a key important
    uint32_t tmem;
    int n_near;
};

__device__ __forceinline__ uint64_t tc_operand(uint32_t addr) {          // K-major rows of 128 bytes, 128-byte swizzle, eight rows = 1 KB
    return (uint64_t)((addr >> 4) & 0x3fffu) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// d (+)= rows x keys over all channels: [128 rows] x [64 keys], bf16 operands, fp32 accumulators
template <int D>
__device__ __forceinline__ void tc_product(uint32_t d, uint32_t rows, uint32_t keys, bool add) {
    using S = TcShape<D>;
    constexpr uint32_t kShape = (1u << 4) | (1u << 7) | (1u << 10) | ((kTcKeys >> 3) << 17) | ((kTcRows >> 4) << 24);
    const uint64_t a = tc_operand(rows), b = tc_operand(keys);
#pragma unroll
    for (int kk = 0; kk < S::kSteps; ++kk) {
        const uint64_t da = a + ((kk >> 2) * S::kRowBlock + (kk & 3) * 32) / 16, db = b + ((kk >> 2) * S::kKeyBlock + (kk & 3) * 32) / 16;
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                     ::"r"(d), "l"(da), "l"(db), "r"(kShape), "r"((uint32_t)(add || kk)) : "memory");
    }
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_load8(uint32_t (&v)[8], uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(addr));
}
__device__ __forceinline__ void tc_wait_loads() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// the values are there behind it
__device__ __forceinline__ void tc_loaded(uint32_t (&v)[8]) {
    asm volatile("" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]));
}
// the eight warps that work on rows and keys, without the one that issues products
__device__ __forceinline__ void tc_sync() { asm volatile("barrier.cta.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void tc_arrive(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory"); }
__device__ __forceinline__ void tc_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// all 512 columns, by one warp (a block of this kernel has an SM to itself: kTcMinSmem)
__device__ __forceinline__ void tc_alloc(uint32_t dst) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(dst) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tc_free(uint32_t tmem) { asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem)); }

// error of a logit of phase A (before the 1/sqrt(d)) per unit of the unit's largest key magnitude; n1, n2, n3: 1-norms of the
// row and of its second and third pieces (see the head of the file). k2.q3 and r2.q3 are left out; adding the small parts
// together and scaling rounds twice. The small products share an accumulator over all channels, so the bound is up to 1.9 times
// split_error's, but phase B's own, with 17 roundings per 16 terms, is narrower: logits formed again, here / mma.sync, 32 units x
// 8192 keys, G 4, w 128, 47982 / 47999 of 1.3e8, 128 x 3390, w 256, 37480 / 37934, one key channel 64 times the others 986301 / 1115750.
__device__ __forceinline__ float tc_split_error(float n1, float n2, float n3) {
    return 2.0267e-6f * (8.f * n1 * (1.f / 8192.f) + 16.f * n2 * (1.f / 8192.f) + 24.f * n3) * 1.05f +
           1.3e-7f * (n2 * (1.f / 64.f) + n1 * (1.f / 8192.f) + n3) + n3 * (1.f / 60.f);
}

// exp(s / sqrt(D)) is added to z: 2^(n / 16) from a table, a Taylor polynomial of degree 6 on what is left (at most ln2 / 32:
// truncation 5e-16), the 1/sqrt(D) inside the constants. An s beyond the limit gives any number or none; a logit that is not
// `on` may lie there and adds nothing: its power of two is that of n = 0 (0 x infinity would be no number).
template <int D> struct TcExp {
    static constexpr double kScale = D == 128 ? 2.040278893193579 : 2.8853900817779268;
    static constexpr double kC1 = D == 128 ? 0.49012907172436826 : 0.3465735902718734;              // sqrt(D) ln2 / 16, its first 35 bits
    static constexpr double kC2 = D == 128 ? 9.905336546228511e-12 : 8.09925509332828e-12;
    static constexpr double c1 = D == 128 ? inv_root_dim(128) : 0.125;
    static __device__ __forceinline__ double entry(int i) {
        const double e = exp2((double)i / 16.0);
        return __hiloint2double(__double2hiint(e) - (i << 16), __double2loint(e));
    }
    static __device__ __forceinline__ void add(double& z, double s, const double* exp16, bool on) {
        constexpr double kMagic = 6755399441055744.0;
        const double t = fma(s, kScale, kMagic), nf = t - kMagic;
        const int n = on ? __double2loint(t) : 0;
        const double r = fma(nf, -kC2, fma(nf, -kC1, s));
        double p = c1 * c1 * c1 * c1 * c1 * c1 / 720.0;
        p = fma(p, r, c1 * c1 * c1 * c1 * c1 / 120.0);
        p = fma(p, r, c1 * c1 * c1 * c1 / 24.0);
        p = fma(p, r, c1 * c1 * c1 / 6.0);
        p = fma(p, r, c1 * c1 / 2.0);
        p = fma(p, r, c1);
        p = fma(p, r, 1.0);
        const double e = exp16[n & 15];                       // n << 16 = (n >> 4) << 20 for the exponent and what the table has less
        z = fma(on ? p : 0.0, __hiloint2double(__double2hiint(e) + n * 65536, __double2loint(e)), z);
    }
};

// The block's keys in tiles of 64, each thread's part of a tile in registers on its way to shared memory: warp w brings keys
// 8 w .. 8 w + 7.
template <int D> struct TcKeys {
    using S = TcShape<D>;
    const bf16_t* keys;                          // the block's first
    int n_keys;
    uint4 raw[S::kLoads];
    __device__ __forceinline__ int row(int i) const {                    // of the tile
        const int lane = threadIdx.x & 31, per = D / 8;
        return (threadIdx.x >> 5) * 8 + i * (32 / per) + lane / per;
    }
    __device__ __forceinline__ int chunk() const { return (threadIdx.x & 31) % (D / 8); }
    __device__ __forceinline__ uint32_t place(int i) const {             // of the thread's i-th 16 bytes inside an operand
        const int r = row(i), c = chunk();
        return (c >> 3) * S::kKeyBlock + r * 128 + (((c & 7) ^ (r & 7)) << 4);
    }
    __device__ __forceinline__ void load(int tile) {
#pragma unroll
        for (int i = 0; i < S::kLoads; ++i) {
            const int j = tile * kTcKeys + row(i);
            raw[i] = j < n_keys ? __ldg(reinterpret_cast<const uint4*>(keys + (size_t)j * D) + chunk()) : make_uint4(0, 0, 0, 0);
        }
    }
    __device__ __forceinline__ uint32_t amax() const {                   // bf16 bits, of the warp's eight keys
        uint32_t m = 0u;
#pragma unroll
        for (int i = 0; i < S::kLoads; ++i)
            m = max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(m, raw[i].x), raw[i].y), raw[i].z), raw[i].w);
        return __reduce_max_sync(0xffffffffu, max(m & 0xffffu, m >> 16));
    }
    // (phase B) the values as they are, asynchronously, and their magnitude
    __device__ __forceinline__ void copy(unsigned char* at, int tile) const {
#pragma unroll
        for (int i = 0; i < S::kLoads; ++i) {
            const int j = tile * kTcKeys + row(i);
            cp_async16_zfill(smem_addr(at + place(i)), reinterpret_cast<const uint4*>(keys + (size_t)(j < n_keys ? j : 0) * D) + chunk(), j < n_keys);
        }
    }
    __device__ __forceinline__ uint32_t amax(const unsigned char* at) {
#pragma unroll
        for (int i = 0; i < S::kLoads; ++i) raw[i] = *reinterpret_cast<const uint4*>(at + place(i));
        return amax();
    }
    __device__ __forceinline__ void store_pieces(unsigned char* at, SplitGrid g) const {
#pragma unroll
        for (int i = 0; i < S::kLoads; ++i) {
            const uint32_t a[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
            uint32_t k1[4], k2[4], r2[4];
            split_key(a, g, k1, k2, r2);
            unsigned char* dst = at + place(i);
            *reinterpret_cast<uint4*>(dst) = make_uint4(k1[0], k1[1], k1[2], k1[3]);
            *reinterpret_cast<uint4*>(dst + S::kKeyPiece) = make_uint4(k2[0], k2[1], k2[2], k2[3]);
            *reinterpret_cast<uint4*>(dst + 2 * S::kKeyPiece) = make_uint4(r2[0], r2[1], r2[2], r2[3]);
        }
    }
};

// A group's rows as operands, two threads to a row: their pieces (and norms), or their raw values. Returns false if a row
// leaves the safe range.
template <int D, bool kPieces>
__device__ __forceinline__ bool tc_store_rows(const PcRows& R, const bf16_t* Qu, int row0, unsigned char* at, float* n1_sm, float* qe_sm) {
    using S = TcShape<D>;
    constexpr int kN = D / 16;                                // 16-byte pieces of half a row
    const int r = threadIdx.x >> 1, half = threadIdx.x & 1, row = row0 + r;
    const bool on = R.pos(row) > 0;
    uint4 raw[kN];
    const uint4* src = reinterpret_cast<const uint4*>(R.q<bf16_t, D>(Qu, on ? row : R.rows - 1)) + half * kN;
#pragma unroll
    for (int i = 0; i < kN; ++i) raw[i] = on ? __ldg(src + i) : make_uint4(0, 0, 0, 0);
    auto place = [&](int i) {
        const int c = half * kN + i;
        return at + (c >> 3) * S::kRowBlock + r * 128 + (((c & 7) ^ (r & 7)) << 4);
    };
    if constexpr (!kPieces) {
#pragma unroll
        for (int i = 0; i < kN; ++i) *reinterpret_cast<uint4*>(place(i)) = raw[i];
        return true;
    }
    uint32_t mx = 0u;
#pragma unroll
    for (int i = 0; i < kN; ++i)
        mx = max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(mx, raw[i].x), raw[i].y), raw[i].z), raw[i].w);
    uint32_t m16 = max(mx & 0xffffu, mx >> 16);
    m16 = max(m16, __shfl_xor_sync(0xffffffffu, m16, 1));
    const bool ok = m16 < kSplitMaxBits;
    const float c = split_query_const(ok ? __uint_as_float(m16 << 16) : 1.f);
    float n1 = 0.f, n2 = 0.f, n3 = 0.f;
#pragma unroll
    for (int i = 0; i < kN; ++i) {
        const uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
        uint32_t p[3][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float a[2] = {__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u)};
            float x1[2], x2[2], x3[2];
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                split_query(a[y], c, x1[y], x2[y], x3[y]);
                n1 += fabsf(a[y]); n2 += fabsf(x2[y]); n3 += fabsf(x3[y]);
            }
            auto pack = [](const float (&x)[2]) { return (__float_as_uint(x[0]) >> 16) | (__float_as_uint(x[1]) & 0xffff0000u); };   // exact: bf16 numbers
            p[0][e] = pack(x1); p[1][e] = pack(x2); p[2][e] = pack(x3);
        }
#pragma unroll
        for (int y = 0; y < 3; ++y) *reinterpret_cast<uint4*>(place(i) + y * S::kRowPiece) = make_uint4(p[y][0], p[y][1], p[y][2], p[y][3]);
    }
    n1 += __shfl_xor_sync(0xffffffffu, n1, 1);
    n2 += __shfl_xor_sync(0xffffffffu, n2, 1);
    n3 += __shfl_xor_sync(0xffffffffu, n3, 1);
    if (half == 0 && row < (R.rows + 7) / 8 * 8) {
        n1_sm[row] = n1 * 1.0001f;
        qe_sm[row] = tc_split_error(n1, n2, n3) * 1.0001f;
    }
    return ok;
}

struct TcBlock {                                 // what both phases know of the block
    PcRows R;
    const bf16_t *Qu, *Ku;
    int k_begin, k_end, n_keys;
    unsigned char* operands;
    TcMisc* tc;
    uint32_t tmem;
    int step;                                    // tiles so far: buffers alternate, their barriers' phases every second time
    bool late;                                   // a wait expired (the others are skipped)
    __device__ __forceinline__ void wait(int at) {
        if (!late && !mbar_wait(smem_addr(tc->bar + (at & 1)), (at >> 1) & 1)) late = true;
        tc_after_sync();
    }
};

// ---- phase A: sums of exp(s) per row into zs ----
// The ninth warp: starts a tile's products when all warps have stored their pieces of it.
template <int D>
__device__ __noinline__ void tc_issue_a(const TcBlock B) {
    using S = TcShape<D>;
    const int n_tiles = (B.n_keys + kTcKeys - 1) / kTcKeys, n = n_tiles * ((B.R.rows + kTcRows - 1) / kTcRows);
    const uint32_t q1 = smem_addr(B.operands), q2 = q1 + S::kRowPiece, q3 = q2 + S::kRowPiece;
    if ((threadIdx.x & 31) == 0)
        for (int i = 0; i < n; ++i) {
            const int s = i & 1;
            if (!mbar_wait(smem_addr(B.tc->full + s), (i >> 1) & 1)) break;      // (the others' waits expire too)
            tc_after_sync();
            const uint32_t k1 = q3 + S::kRowPiece + s * S::kStage, k2 = k1 + S::kKeyPiece, r2 = k2 + S::kKeyPiece, d = B.tmem + s * 256;
            tc_product<D>(d, q1, k1, false);
            tc_product<D>(d + 64, q2, k1, false);
            tc_product<D>(d + 64, q1, k2, true);
            tc_product<D>(d + 128, q2, k2, false);
            tc_product<D>(d + 192, q3, k1, false);
            tc_product<D>(d + 192, q2, r2, true);
            tc_product<D>(d + 192, q1, r2, true);
            tc_commit(smem_addr(B.tc->bar + s));
        }
    __syncwarp();
}

// The eight warps. Returns false if a row or a logit leaves the range.
template <int D>
__device__ __noinline__ bool tc_phase_a(TcBlock& block, double* zs, float* n1_sm, float* qe_sm, uint32_t* amax) {
    using S = TcShape<D>;
    TcBlock B = block;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, half = warp >> 2, my = (warp & 3) * 32 + lane;
    const int n_tiles = (B.n_keys + kTcKeys - 1) / kTcKeys, first_cut = B.R.P - B.R.w + 1;        // keys from here on are not every row's
    unsigned char* const keys_sm = B.operands + 3 * S::kRowPiece;
    const double* const exp16 = B.tc->exp16;
    TcKeys<D> keys{B.Ku + (size_t)B.k_begin * D, B.n_keys, {}};
    bool ok = true;
    float top = 0.f;
    uint32_t am_all = 0u;
    for (int row0 = 0, turn = 0; row0 < B.R.rows; row0 += kTcRows, turn ^= 1) {
        keys.load(0);
        // (the group before is done with the rows' pieces: every warp has waited for its last tile)
        ok &= tc_store_rows<D, true>(B.R, B.Qu, row0, B.operands, n1_sm, qe_sm);
        const int qpos = B.R.pos(row0 + my);
        double z = 0.0;
        auto cut = [&](int c) {                               // the warp's keys of tile c to its buffer, which tile c - 2 is done with
            const int s = (B.step + c) & 1;
            const uint32_t am = keys.amax();
            am_all = max(am_all, am);
            keys.store_pieces(keys_sm + s * S::kStage, split_grid(am));
            fence_async_smem();
            tc_before_sync();
            __syncwarp();
            if (lane == 0) tc_arrive(smem_addr(B.tc->full + s));
        };
        if (n_tiles) {
            cut(0);
            keys.load(1);
        }
        for (int c = 0; c < n_tiles; ++c) {
            if (c + 1 < n_tiles) {
                cut(c + 1);
                if (c + 2 < n_tiles) keys.load(c + 2);
            }
            B.wait(B.step + c);
            const uint32_t from = B.tmem + ((uint32_t)((warp & 3) * 32) << 16) + ((B.step + c) & 1) * 256 + half * 32;
            const int j0 = B.k_begin + c * kTcKeys + half * 32;
            const bool last = j0 + 32 > B.k_end || j0 + 32 > first_cut;
            // (integer instructions issue at half rate like fp64: what only the last keys need is kept out of the others)
            auto sums = [&](auto masked) {
                uint32_t a[2][4][8];
                auto fetch = [&](int g) {
#pragma unroll
                    for (int x = 0; x < 4; ++x) tc_load8(a[g & 1][x], from + x * 64 + g * 8);
                };
                fetch(0);
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    tc_wait_loads();
#pragma unroll
                    for (int x = 0; x < 4; ++x) tc_loaded(a[g & 1][x]);
                    if (g < 3) fetch(g + 1);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const uint32_t(&v)[4][8] = a[g & 1];
                        const float hi = __uint_as_float(v[0][k]), mid = __uint_as_float(v[1][k]), small = __uint_as_float(v[2][k]) + __uint_as_float(v[3][k]);
                        bool on = true;
                        if constexpr (decltype(masked)::value) {               // causal row: keys 1..position of the query
                            const int j = j0 + g * 8 + k;
                            on = j < B.k_end && j < qpos;
                        }
                        if (on) top = fmaxf(top, fabsf(hi + mid));
                        TcExp<D>::add(z, ((double)hi + (double)mid) + (double)small, exp16, on);
                    }
                }
            };
            if (last) sums(std::true_type()); else sums(std::false_type());
        }
        B.step += n_tiles;
        B.tc->z[turn][half][my] = z;
        tc_sync();
        if (tid < kTcRows && row0 + tid < B.R.rows) zs[row0 + tid] = B.tc->z[turn][0][tid] + B.tc->z[turn][1][tid];
    }
    tc_before_sync();
    if (lane == 0) atomicMax(amax, am_all);
    block.step = B.step; block.late = B.late;
    return ok && top < (float)(kPcLogitLimit * (D == 128 ? 11.3137 : 8.0));
}

// The listed logits, four lanes each: what is sure to be important is joined to the key's register, what is within the
// threshold's own error is left to the exact rows.
template <int D>
__device__ __noinline__ void tc_near(const PromptParams& p, const TcBlock B, const uint32_t* list, int n, const double* thr_sm, const float* qe_sm,
                                     double eps_unit, uint32_t* words_g, uint32_t* flags, PcMisc* misc) {
    const int sub = threadIdx.x & 3;
    for (int i0 = (threadIdx.x >> 5) * 8; i0 < n; i0 += kPcWarps * 8) {
        const int i = i0 + ((threadIdx.x & 31) >> 2);
        const bool on = i < n;
        const uint32_t x = list[on ? i : i0];
        const int row = (int)(x >> 20), j = B.k_begin + (int)(x & 0xfffffu);
        QuadRow<bf16_t, D> q;
        q.load(B.R.q<bf16_t, D>(B.Qu, row), sub);
        const bf16_t* const rows[1] = {B.Ku + (size_t)j * D};
        double s[1];
        quad_exact_dots<bf16_t, D, 1>(q, rows, sub, s);
        const double th = thr_sm[row], margin = s[0] * inv_root_dim(D) - th, e = eps_unit * (double)qe_sm[row] + 1e-13 * (1.0 + fabs(th));
        if (on && sub == 0) {
            const uint32_t mark = pc_mark(p.w, B.R.rho(row), B.R.pos(row));
            if (margin > e) { if (p.w <= 32) atomicOr(words_g + j, mark); else atomicMax(words_g + j, mark); }
            else if (margin >= -e) pc_leave_open(flags, misc, row, j);
        }
    }
    if (threadIdx.x == 0) atomicAdd(p.counters + CNT_NEAR, (unsigned long long)n);
}

// ---- phase B: verdicts of the block's keys for every row -> scratch registers ----
template <int D>
__device__ __noinline__ void tc_phase_b(const PromptParams& p, TcBlock& block, const double* thr_sm, const float* n1_sm, const float* qe_sm, double eps_unit,
                                        uint32_t* words_g, uint32_t* flags, PcMisc* misc) {
    using S = TcShape<D>;
    TcBlock B = block;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, half = warp >> 2, my = (warp & 3) * 32 + lane;
    const int n_tiles = (B.n_keys + kTcKeys - 1) / kTcKeys;
    const uint32_t rows_at = smem_addr(B.operands), keys_at = rows_at + S::kRowPiece;
    unsigned char* const keys_sm = B.operands + S::kRowPiece;             // the tiles' stages, then the list
    uint32_t* const list = reinterpret_cast<uint32_t*>(keys_sm + kTcStagesB * S::kKeyPiece);
    static_assert(S::kRowPiece + kTcStagesB * S::kKeyPiece + kTcNearCap * 4 <= S::kOperands, "the list fits behind the operands");
    const double root_d = D == 128 ? 11.313708498984760390 : 8.0;
    const int log2g = B.R.log2g;
    TcKeys<D> keys{B.Ku + (size_t)B.k_begin * D, B.n_keys, {}};
    auto fetch = [&](int c) {                                 // tile c on its way to its stage, whose tile is done with
        if (c < n_tiles) keys.copy(keys_sm + (c % kTcStagesB) * S::kKeyPiece, c);
        cp_async_commit();
    };
    if (tid < 2 * kTcKeys) B.tc->words[0][tid] = 0u;
    if (tid == 0) B.tc->n_near = 0;
    bool flush = false;
    for (int row0 = 0; row0 < B.R.rows; row0 += kTcRows) {
        __syncthreads();                                      // thresholds are there; everybody is done with the group before
#pragma unroll
        for (int c = 0; c < kTcStagesB; ++c) fetch(c);
        tc_store_rows<D, false>(B.R, B.Qu, row0, B.operands, nullptr, nullptr);
        const int row = row0 + my, qpos = B.R.pos(row);
        const float tf = qpos ? (float)(thr_sm[row] * root_d) : INFINITY;
        // a chain of D / 16 steps of 17 roundings of 2^-23 on sums of at most A |q|_1 (a tenth of slack), the threshold's own
        // rounding, and the threshold's error
        const float err_a = qpos ? (float)p.bound_scale * ((float)(D / 16 * 17) * 1.1f / 8388608.f * n1_sm[row]) : 0.f;
        const float slack = qpos ? (tf > -3e38f && tf < 3e38f ? fabsf(tf) : 0.f) * 2.4e-7f + (float)(eps_unit * qe_sm[row] * root_d) * 1.01f : 0.f;
        auto bring = [&](int c) {
            const int s = (B.step + c) & 1, stage = c % kTcStagesB;
            cp_async_wait<2>();
            const uint32_t am = keys.amax(keys_sm + stage * S::kKeyPiece);       // (of the thread's own copies)
            if (lane == 0) B.tc->scale[stage][warp] = split_amax(am);
            fence_async_smem();
            tc_before_sync();
            const bool full = __syncthreads_or(flush);
            if (warp == (c & 7) && lane == 0) {
                tc_after_sync();
                tc_product<D>(B.tmem + s * 64, rows_at, keys_at + stage * S::kKeyPiece, false);
                tc_commit(smem_addr(B.tc->bar + s));
            }
            return full;
        };
        auto settle = [&](int c, bool full) {                 // tile c's registers, and the list if it is long (behind a barrier)
            const int s = (B.step + c) & 1, at = c * kTcKeys + tid;
            if (tid < kTcKeys) {
                const uint32_t word = B.tc->words[s][tid];
                B.tc->words[s][tid] = 0u;
                if (at < B.n_keys) words_g[B.k_begin + at] = row0 ? pc_join(p.w, __ldcg(words_g + B.k_begin + at), word) : word;
            }
            if (full) {                                       // uniform
                __syncthreads();
                tc_near<D>(p, B, list, B.tc->n_near, thr_sm, qe_sm, eps_unit, words_g, flags, misc);
                __syncthreads();
                if (tid == 0) B.tc->n_near = 0;
                __syncthreads();
                flush = false;
            }
        };
        if (n_tiles) bring(0);
        for (int c = 0; c < n_tiles; ++c) {
            bool full = false;
            if (c + 1 < n_tiles) {
                full = bring(c + 1);
                if (c) settle(c - 1, full);
            } else if (c) {
                full = __syncthreads_or(flush);
                settle(c - 1, full);
            }
            B.wait(B.step + c);
            const int s = (B.step + c) & 1, j0 = B.k_begin + c * kTcKeys + half * 32;
            const uint32_t from = B.tmem + ((uint32_t)((warp & 3) * 32) << 16) + s * 64 + half * 32;
            uint32_t near = 0u;                               // keys of this row to be formed again
            uint32_t a[4][8];
#pragma unroll
            for (int g = 0; g < 4; ++g) tc_load8(a[g], from + g * 8);
            tc_wait_loads();
            auto judge = [&](auto masked) {
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    tc_loaded(a[g]);
                    const float err = fmaf(err_a, B.tc->scale[c % kTcStagesB][half * 4 + g], slack), above = tf + err, below = tf - err;
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float x = __uint_as_float(a[g][k]);
                        bool on = true;
                        if constexpr (decltype(masked)::value) {
                            const int j = j0 + g * 8 + k;
                            on = j < B.k_end && j < qpos;
                        }
                        const bool sure = on && x >= above;
                        const uint32_t who = __ballot_sync(0xffffffffu, sure);
                        if (lane == 0) B.tc->who[warp][g * 8 + k] = who;
                        if (on && !sure && !(x <= below)) near |= 1u << (g * 8 + k);
                    }
                }
            };
            if (j0 + 32 > B.k_end || j0 + 32 > B.R.P - B.R.w + 1 || row0 + kTcRows > B.R.rows) judge(std::true_type()); else judge(std::false_type());
            __syncwarp();
            const uint32_t mine = B.tc->who[warp][lane];      // rows that find key j0 + lane important
            __syncwarp();
            fetch(c + kTcStagesB);
            const int r0 = row0 + (warp & 3) * 32;
            if (mine) {
                uint32_t mark = 0u;
                if (p.w > 32) {                               // the latest query
                    mark = pc_mark(p.w, 0, B.R.pos(r0 + 31 - __clz(mine)));
                } else {
                    for (int x = 0; x < 32; x += 1 << log2g)
                        if ((mine >> x) & ((1u << (1 << log2g)) - 1u)) mark |= pc_mark(p.w, B.R.rho(r0 + x), 0);
                }
                if (p.w <= 32) atomicOr(&B.tc->words[s][half * 32 + lane], mark);
                else atomicMax(&B.tc->words[s][half * 32 + lane], mark);
            }
            for (; near; near &= near - 1u) {
                const int at = atomicAdd(&B.tc->n_near, 1);
                if (at < kTcNearCap) list[at] = ((uint32_t)row << 20) | (uint32_t)(c * kTcKeys + half * 32 + __ffs(near) - 1);
                flush |= at >= kTcNearFlush;
            }
        }
        if (n_tiles) {
            __syncthreads();
            settle(n_tiles - 1, true);
        }
        B.step += n_tiles;
        tc_before_sync();
    }
    block.late = B.late;
    __syncthreads();
}

template <int D>
__host__ __device__ inline PcSmem tc_smem_layout(int rows8) {
    using S = TcShape<D>;
    PcSmem s{};
    int off = 0;
    auto take = [&](int bytes) { int at = off; off = (off + bytes + 127) / 128 * 128; return at; };
    s.ring = take(S::kOperands);
    s.frag = kPcKeys * D * 2 + kPcWarps * kTcRowRoom * 4 * D * 8;        // (of pc_fp64_rows: registers behind its keys and rows)
    static_assert(kPcKeys * D * 2 + kPcWarps * kTcRowRoom * 4 * D * 8 + kPcKeys * 4 <= S::kOperands, "all three fit the operands");
    s.zs = take((rows8 > 64 ? rows8 : 64) * 8);
    s.thr = take(rows8 * 8);
    s.n1 = take(rows8 * 4);
    s.qe = take(rows8 * 4);
    s.flags = take((rows8 + 31) / 32 * 4);
    s.list = take(kPcWarps * 32);
    s.misc = take((int)sizeof(PcMisc));
    s.tc = take((int)sizeof(TcMisc));
    s.total = off > kTcMinSmem ? off : kTcMinSmem;
    return s;
}

}  // namespace corm
