// Decode step: one launch, a thread-block cluster per unit, any dtype, head_dim and group size.
//
// The cluster's blocks share the unit's live slots (whole 32-slot words each) and do the whole of Algorithm 1:
//   1. every warp streams 16-key tiles of K and V through its own ring of shared-memory stages (2-D tensor-map copies
//      with the 128-byte swizzle, mbarriers, bounded waits): logits, probabilities, P.V; no block-wide step in the loop;
//   -- the warps push {m, Z} per head to all blocks: log-sum-exp, thresholds; the blocks push their output numerators to the
//      block that writes them
//   2. verdicts of the block's slots, register update, keep bits;
//   -- the warps push their counts of kept slots, and keep bits and registers of the unit's last words: new length, places of
//      holes and movers
//   3. hole filling, shared over the cluster; the first block publishes the unit's new length.
//
// bf16 logits on the tensor cores (corm_mma.cuh): keys cut into pieces k1, k2, r2, queries into q1, q2, q3. An
// mma.m16n8k16 has eight columns, so the pieces of several heads share one: for a group of up to four heads the columns
// are (q1, q2) of each, and the accumulators of different columns are different numbers, so every product of pieces is
// summed apart (exactly, where the pieces allow). Per 16 keys and 16 channels: 3 mma for one or two heads (the q3's take
// the other columns), 5 for four, 8 for eight. P.V on the tensor cores as well: A = V^T (ldmatrix.trans), B = the
// probabilities, each fp32 number as three bf16 whose sum it is (24 bits = 8 + 8 + 8): of one or two heads they fill the
// eight columns of one mma, of four heads two, of eight three. Two parts leave 2^-18 of a probability out, which showed:
// outputs that are not the exact ones rounded to bf16, of 10^4: two parts 9-12, three 1 (one to eight heads, 64 and 128
// channels), as with fp32 products on the CUDA cores.
// fp32: a key per lane (its channels shared by two half-warps), fp64 products on the CUDA cores, P.V by fp32 FMAs. A bf16
// unit with a key or query element the pieces cannot hold (2^56 and more, infinity, NaN) takes that loop too: its products
// have no bounds on the tensor cores. So does one whose bounds are too wide to be of use (kDcReach).
//
// What bounds it: on units of a few hundred keys the chain of round trips (8 units x 170 keys, fp32, at 9.4 us a step:
// launch and length 2.0, first tiles 1.8, pushes and thresholds 1.5, verdicts 0.8, counts and lists 1.6, moves 1.5), in part
// instructions that are not in the cache yet (ncu: 1.8 warps of 8.9 wait for them per issue); on long units instruction issue in the streaming loop: about
// 650 instructions per tile (192 of them the two-element additions that cut the keys), of 5000 cycles per tile and warp
// with 16 warps on an SM only 270 are spent waiting for its copies. So one stage each for K and V is enough (with two for
// K: 32 units x 8200 keys 43 us a step instead of 38), and what is smaller leaves more L1. Units differ in length and SMs
// hold one block or two, which is what keeps the rest of HBM's rate away.
// Measured, us per step from one call per step, before -> first version -> before the pushes (now: below):
//   64 units x 970 keys, G 8, bf16          253 -> 32 -> 27     128 units x 1090 keys, G 4, 64 channels   143 -> 30 -> 26
//   20 units x 250 keys, G 2, fp32           64 -> 16 -> 13     8 units x 170 keys, G 1, fp32            37.7 -> 14 -> 11
//   128 units x 2800 keys, G 4, bf16         86 -> 68 -> 54     32 units x 21400 keys, G 4, bf16          133 -> 103 -> 80
//   32 units x 8200 keys, G 4, no eviction   55 -> 47 -> 38     32 units x 1160 keys, G 1, bf16            35 -> 24 -> 20
// (from one warp per key and the last-arriving split finishing the unit, from fp64 logits on the CUDA cores with every
// block an equal share of all tiles and a second launch for the verdicts, from the block-per-split kernel).
//
// What the blocks tell one another is pushed (st.async: value and byte count travel together, one way), each block waiting on
// its own barriers, instead of cluster barriers and loads from the peers behind them (two round trips and a flush each). A push
// orders nothing but itself, so whatever one block needs of another's is in a push (or, where heads are formed again or lists go
// to scratch, behind a meeting with release and acquire). us per request, cluster barriers -> pushes: one fp32 sequence, 64
// steps, 767 -> 677; 32 layers 12260 -> 10690; G 8 1490 -> 1400; 64 channels 1536 -> 1400; fp32 G 2 815 -> 720; G 4, 128 units x
// 1800 keys 5980 -> 5880, paged and chained 6130 -> 6140.
//
// Verdicts are the fp64 ones: a slot's logit is kept in fp32, and one that lies within the proven error of its threshold
// is formed again in fp64. If it then lies within the error of the log-sum-exp itself, the head is marked and the
// cluster forms that head's log-sum-exp and verdicts in fp64 once more before anything is evicted (rare).
#pragma once

#include <cuda.h>

#include "corm_fast.cuh"
#include "corm_mma.cuh"

namespace corm {

constexpr int kDcMaxCluster = 8;
constexpr int kDcKeys = 16;                       // keys per tile

struct DecodeClusterParams {
    DecodeParams p;
    int32_t G;
    int32_t lcap;                                 // logits that fit on chip, per block (a longer block's go to p.stash)
    float bound_scale;
};

template <typename T, int D, int GP> struct DcShape {
    static constexpr bool kBf16 = Elem<T>::kBytes == 2;
    static constexpr int kRow = D * Elem<T>::kBytes;
    static constexpr int kBoxes = kRow / 128;     // 128-byte wide boxes of the swizzled copies
    static constexpr int kBox = kDcKeys * 128;
    static constexpr int kTile = kDcKeys * kRow;
    static constexpr int kKs = kTile >= 4096 ? 1 : 2;
    static constexpr int kVs = kTile >= 4096 ? 1 : 2;
    static constexpr int kStages = kKs + kVs;
    static constexpr int kPieces = GP == 8 ? 6 : GP == 4 ? 4 : 2;   // words per lane and 16 channels of the query pieces
    static constexpr int kWarpRing = kStages * kTile;
    static constexpr int kProb = kBf16 ? kDcKeys * (GP == 8 ? 48 : GP == 4 ? 32 : 16) : kDcKeys * GP * 4;   // a warp's probabilities
};
// resident blocks per SM the register budget is set for
template <typename T, int D, int GP, int NW> __host__ __device__ constexpr int dc_blocks() {
    return Elem<T>::kBytes == 4 ? (D == 128 ? 12 : 16) / NW : (GP == 8 ? 12 : 16) / NW;
}

// Slots a step may evict from a unit for its moves to be listed on chip: what moves lies in the unit's last 32 words then.
constexpr int kDcListCap = 992;

// What the ring holds once the tiles are done: the warps' records at the start of their parts, and from 4 KB on the keep bits
// of the block's words and, behind them, the lists of a step with few moves or the prefix sums (one more than words) of a
// step with many. So the words a block may own follow from the instance's ring: 4096 for the rings of 64 KB, 3583 for the
// 32 KB of fp32 / 64 channels. The ring's last 4 KB hold the registers of the unit's last 32 words.
constexpr int kDcRecBytes = 4096, kDcRegBytes = 32 * 32 * 4;
template <typename T, int D, int GP, int NW> __host__ __device__ constexpr int dc_max_words() {
    constexpr int n = (NW * DcShape<T, D, GP>::kWarpRing - kDcRecBytes - 4) / 8;
    return n < 4096 ? n : 4096;
}
template <typename T, int D, int GP, int NW> __host__ __device__ constexpr bool dc_ring_holds_lists() {
    constexpr int words = dc_max_words<T, D, GP, NW>(), lists = 2 * kDcListCap * 4, sums = 4 * (words + 1);
    constexpr int ring = DcShape<T, D, GP>::kWarpRing;
    return GP * D * 4 <= kDcRecBytes && kDcRecBytes + kDcRegBytes <= ring && kDcRecBytes + 4 * words + sums <= NW * ring &&
           kDcRecBytes + 4 * words + lists + kDcRegBytes <= NW * ring;
}

constexpr int kDcOpenCap = 32;
// A block's barriers: what every warp of the unit's blocks found (kDcRecords), the block's share of the outputs' numerators
// from every block (kDcOutputs), the warps' verdicts in numbers, the unit's last keep bits and registers and the appended row
// (kDcCounts), all blocks (kDcMeet) and, at the first block, the others being done with the unit (kDcDone).
enum { kDcRecords = 0, kDcOutputs = 1, kDcCounts = 2, kDcMeet = 3, kDcDone = 4, kDcBars = 5 };
template <int NW, int GP> struct DcMisc {
    unsigned long long bar[kDcBars], stamp;
    // pushed by the unit's blocks, block by block and warp by warp: {m, Z} of each head, state words, verdicts (kept slots |
    // heads to be formed exactly << 24, important keys), and the keep bits of the unit's last 32 words, the last one first
    struct alignas(16) Entry { double m, z; };
    union { Entry rec[GP][kDcMaxCluster * NW]; int scan[NW * 32]; };    // (the scan: of steps with many moves)
    uint2 verdicts[kDcMaxCluster * NW];
    uint32_t tail[32];
    // largest key magnitude (bf16 bits), 1 << 16 if the block took the fp64 loop for it, 1 << 17 if a wait expired, 1 << 18
    // if the unit cannot take the token
    uint32_t state[kDcMaxCluster * NW];
    double thr[GP], Zt[GP], log_t;
    double red[NW][2], mz[2];                     // exact heads
    float sc[GP][NW], qe[GP], thr_f[GP], slack[GP];
    float qe_part[NW][GP];                        // the warps' shares of qe
    uint32_t cut_for;                             // bf16: the unit's magnitude before the appended key; 0 if that asks for the fp64 loop
    uint32_t flags[NW];                           // per warp: heads to be formed exactly
    struct alignas(16) Counts { int count, n_imp, pad[2]; } cnt;      // kept slots and important keys of the block (exact heads)
    int n_open;                                   // open verdicts of marked heads: slot << 3 | head
    uint32_t open[kDcOpenCap];
    int n_moved;                                  // row moves of the unit
};

// All blocks of the unit meet: what they wrote before is there for the others behind. Returns false if the wait expired.
__device__ __forceinline__ bool dc_meet(uint32_t bar, int cs, uint32_t& phase) {
    __syncthreads();
    if ((int)threadIdx.x < cs) mbar_arrive_peer(map_rank(bar, threadIdx.x));
    return mbar_wait_cluster(bar, phase++ & 1u);
}

// When a bf16 unit takes the fp64 loop. Errors of the tensor-core logits grow with A Aq, the product of the unit's largest key
// and query magnitudes, while its logits need not (one large key channel next to small query channels). Where the bounds
// leave verdicts open in most steps (about A Aq times the unit's keys, per head), forming heads again costs more than fp64
// does: us per step never / always / a multi-pass fp64 kernel, one key channel 256 times the others: 32 units x 20000 keys,
// G 4, 146 / 126 / 131; 32 units x 8200 keys, G 4, 66 / 57 / 55; 128 units x 3400 keys, G 1, 82 / 54 / 54 (ordinary keys 55 /
// 54 / 54); but 128 units x 2800 keys, G 4, 78 / 82 / 84 and 64 units x 700 keys, G 8, 31 / 51. One and two heads switch
// earlier: their fp64 loop costs 0-5 and 12 % of ordinary steps, that of four 20-55 %. And beyond A Aq = 16384 logits would
// be less exact than fp32 probabilities.
constexpr float kDcReach = 16384.f;
template <int GP> __device__ __forceinline__ float dc_reach_keys(int G) { return GP > 2 ? 6e7f : G == 2 ? 4e6f : 5e5f; }
constexpr uint32_t kDcWide = 1u << 16, kDcExpired = 1u << 17, kDcFull = 1u << 18;

struct DcSmem { int prob, q, pieces, newrow, logits, bars, misc, total; };
template <typename T, int D, int GP, int NW>
__host__ __device__ inline DcSmem dc_smem_layout(int lcap) {
    using S = DcShape<T, D, GP>;
    DcSmem s{};
    int off = NW * S::kWarpRing;
    auto take = [&](int bytes) { int at = off; off = (off + bytes + 127) / 128 * 128; return at; };
    s.prob = take(NW * S::kProb);
    s.q = take(GP * D * (S::kBf16 ? 2 : 8));      // fp32: widened to fp64
    // (or the queries widened to fp64)
    s.pieces = take(S::kBf16 ? (D / 16 * S::kPieces * 128 > GP * D * 8 ? D / 16 * S::kPieces * 128 : GP * D * 8) : 0);
    s.newrow = take(2 * S::kRow);
    s.bars = take(NW * S::kStages * 8);
    s.misc = take((int)sizeof(DcMisc<NW, GP>));
    s.logits = take(lcap * 4);
    s.total = off;
    return s;
}

// The GP (G of them, where an instance serves two group sizes) logits of one slot, stored side by side.
template <int GP, bool kGlobal> __device__ __forceinline__ void load_logits(const float* src, int G, float (&out)[GP]) {
    auto ld1 = [](const float* a) { if constexpr (kGlobal) return __ldcg(a); else return *a; };
    if constexpr (GP % 4 == 0) {
#pragma unroll
        for (int h = 0; h < GP; h += 4) {
            const float4* a = reinterpret_cast<const float4*>(src + h);
            float4 v;
            if constexpr (kGlobal) v = __ldcg(a); else v = *a;
            out[h] = v.x; out[h + 1] = v.y; out[h + 2] = v.z; out[h + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int h = 0; h < GP; ++h) out[h] = h < G ? ld1(src + h) : 0.f;
    }
}

// N contiguous elements of the cache past the L1 (rows move between launches that may overlap)
template <typename T, int N> __device__ __forceinline__ void load_slice_cg(const T* p, float (&out)[N]) {
    if constexpr (Elem<T>::kBytes == 2) {
        uint32_t w[N / 2];
        if constexpr (N == 4) { const uint2 v = __ldcg(reinterpret_cast<const uint2*>(p)); w[0] = v.x; w[1] = v.y; }
        else w[0] = __ldcg(reinterpret_cast<const uint32_t*>(p));
#pragma unroll
        for (int i = 0; i < N / 2; ++i) { out[2 * i] = __uint_as_float(w[i] << 16); out[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
    } else if constexpr (N == 4) {
        const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
        out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
    } else {
        const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
        out[0] = v.x; out[1] = v.y;
    }
}

// the largest of the lanes' numbers (none NaN): of the high words, then of the low words that go with it
__device__ __forceinline__ double warp_max(double x) {
    const long long b = __double_as_longlong(x);
    const unsigned long long o = (unsigned long long)(b ^ ((b >> 63) | (long long)0x8000000000000000ull));
    const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(o >> 32));
    const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(o >> 32) == hi ? (uint32_t)o : 0u);
    const unsigned long long m = ((unsigned long long)hi << 32) | lo;
    return __longlong_as_double((long long)(m >> 63 ? m ^ 0x8000000000000000ull : ~m));
}

// exact q.k of a slot by a whole warp: fp64, before the 1/sqrt(d)
template <typename T, int D>
__device__ __forceinline__ double warp_exact_dot_cg(const T* q, const T* k, int lane) {
    constexpr int NPL = D / 32;
    float a[NPL], b[NPL];
    load_slice<T, NPL>(q + lane * NPL, a);
    load_slice_cg<T, NPL>(k + lane * NPL, b);
    double part = 0.0;
#pragma unroll
    for (int i = 0; i < NPL; ++i) part = fma((double)a[i], (double)b[i], part);
    return warp_sum(part);
}

// The marked heads, exactly, by the whole cluster: their log-sum-exp in fp64 with a running maximum, then the verdicts
// that were left open (misc->open, or every slot of the block where those did not fit). A verdict that was sure before holds for the exact threshold too, so adding importance is enough: the register
// gets its newest bit (or stamp), the keep bit is set. About one step in ten of 32 units x 21000 keys comes here: 16 keys
// per warp at a time instead of 8, and no second pass over the keys, took 100 us of such a step to 20.
template <typename T, int D, int NW, int GP>
__device__ __noinline__ bool dc_exact_heads(const DecodeParams& p, int u, int G, int t, int k_begin, int k_end, uint32_t heads,
                                            uint32_t* keep, DcMisc<NW, GP>* misc, int cs, uint32_t phase) {
    const uint32_t meet = smem_addr(&misc->bar[kDcMeet]);
    bool ok = true;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, sub = lane & 3;
    const int32_t* pt_u = p.page_table ? p.page_table + (size_t)u * p.pt_stride : nullptr;
    const T* Kl = reinterpret_cast<const T*>(p.K);
    const uint32_t mz_addr = smem_addr(misc->mz);
    uint32_t* wordu = p.word + (size_t)u * p.C;
    auto row_of = [&](int j) -> const T* { return Kl + kv_row(pt_u, (size_t)u * p.C, j, p.pool_pages, p.status) * D; };
    int added = 0, added_imp = 0;
    auto add_importance = [&](int j) {
        const uint32_t reg = __ldcg(wordu + j), bit = 1u << (j & 31);
        if (p.w <= 32 ? (reg & 1u) : reg == (uint32_t)t) return;
        wordu[j] = p.w <= 32 ? (reg | 1u) : (uint32_t)t;
        added_imp += 1;
        if (!(atomicOr(keep + ((j - k_begin) >> 5), bit) & bit)) added += 1;
    };
    const int n_open = misc->n_open > kDcOpenCap ? -1 : misc->n_open;
    for (int h = 0; h < G; ++h) {
        if (!((heads >> h) & 1u)) continue;
        const T* q = reinterpret_cast<const T*>(p.q) + ((size_t)u * G + h) * D;
        double m, Z;
        warp_exact_lse<T, D>(q, row_of, k_begin + warp * 16, k_end, NW * 16, m, Z);
        if (lane == 0) { misc->red[warp][0] = m; misc->red[warp][1] = Z; }
        __syncthreads();
        if (tid == 0) {
            double mb = -INFINITY, Zb = 0.0;
            for (int x = 0; x < NW; ++x) mb = fmax(mb, misc->red[x][0]);
            for (int x = 0; x < NW; ++x)
                if (misc->red[x][1] > 0.0) Zb += misc->red[x][1] * exp(misc->red[x][0] - mb);
            misc->mz[0] = mb; misc->mz[1] = Zb;
        }
        ok &= dc_meet(meet, cs, phase);
        double M = -INFINITY, Zt = 0.0;
        for (int x = 0; x < cs; ++x) M = fmax(M, ld_peer_f64(map_rank(mz_addr, x)));
        for (int x = 0; x < cs; ++x) {
            const double z = ld_peer_f64(map_rank(mz_addr + 8, x));
            if (z > 0.0) Zt += z * exp(ld_peer_f64(map_rank(mz_addr, x)) - M);
        }
        const double thr = M + log(Zt) + p.log_alpha - log((double)t);
        QuadRow<T, D> qr;
        qr.load(q, sub);
        const int n = n_open < 0 ? k_end - k_begin : n_open;
        for (int i0 = warp * 8; i0 < n; i0 += NW * 8) {       // eight slots per warp, the same sums as above
            const int i = i0 + (lane >> 2);
            const bool on = i < n && (n_open < 0 || (misc->open[i] & 7u) == (uint32_t)h);
            const int j = on ? (n_open < 0 ? k_begin + i : (int)(misc->open[i] >> 3)) : k_begin;
            const T* const rows[1] = {row_of(j)};
            double s[1];
            quad_exact_dots<T, D, 1>(qr, rows, sub, s);
            if (on && sub == 0 && s[0] * inv_root_dim(D) >= thr) add_importance(j);
        }
        ok &= dc_meet(meet, cs, phase);                       // everybody has read mz; the registers of this head are written
    }
    if (added) atomicAdd(&misc->cnt.count, added);
    if (added_imp) atomicAdd(&misc->cnt.n_imp, added_imp);
    return ok;
}

// Verdicts that the error bounds leave open, by a whole warp: lane's slot j, heads `open`; true where a head is sure to
// find the key important. Heads whose threshold is too close to tell are marked in the warp's misc->flags.
template <typename T, int D, int NW, int GP>
__device__ __noinline__ bool dc_open_verdicts(const DecodeParams& p, int u, int G, int j, uint32_t open, float eps_a, DcMisc<NW, GP>* misc) {
    const int lane = threadIdx.x & 31;
    const int32_t* pt_u = p.page_table ? p.page_table + (size_t)u * p.pt_stride : nullptr;
    bool imp = false;
    uint32_t who = __ballot_sync(0xffffffffu, open != 0u);
    int n_near = 0;
    while (who) {
        const int src = __ffs(who) - 1;
        who &= who - 1u;
        const int js = __shfl_sync(0xffffffffu, j, src);
        uint32_t os = __shfl_sync(0xffffffffu, open, src);
        const size_t row = kv_row(pt_u, (size_t)u * p.C, js, p.pool_pages, p.status);
        while (os) {
            const int h = __ffs(os) - 1;
            os &= os - 1u;
            const double s = warp_exact_dot_cg<T, D>(reinterpret_cast<const T*>(p.q) + ((size_t)u * G + h) * D,
                                                     reinterpret_cast<const T*>(p.K) + row * D, lane) * inv_root_dim(D);
            const double th = misc->thr[h], e = (eps_a > 0.f ? (double)(eps_a * misc->qe[h]) : 0.0) + 1e-13 * (1.0 + fabs(th));
            if (lane == src && s - th > e) imp = true;
            if (lane == 0 && fabs(s - th) <= e) {
                misc->flags[threadIdx.x >> 5] |= 1u << h;
                const int at = atomicAdd(&misc->n_open, 1);
                if (at < kDcOpenCap) misc->open[at] = ((uint32_t)js << 3) | (uint32_t)h;
            }
            ++n_near;
        }
    }
    if (lane == 0) atomicAdd(p.counters + CNT_NEAR, (unsigned long long)n_near);
    return imp;
}

// The tiles of a warp: where they lie, the copies that fetch them, and the repair of the one that holds the appended token
// or the unit's end.
template <typename T, int D, int GP, int NW> struct DcTiles {
    using S = DcShape<T, D, GP>;
    const DecodeParams& p;
    const CUtensorMap &kmap, &vmap;
    const int32_t* pt_u;
    unsigned char *ring, *newrow;
    uint32_t bars;
    int u, l_old, t, k_begin, k_end, my_n, my_page;           // lane i keeps the page entry of the warp's tile i

    __device__ __forceinline__ int first_key(int it) const { return k_begin + ((int)(threadIdx.x >> 5) + it * NW) * kDcKeys; }
    __device__ __forceinline__ int row0(int it) const {       // first row of a tile in the layer's K / V storage (all lanes call)
        const int j = first_key(it);
        if (!pt_u) return (int)((size_t)u * p.C) + j;
        const int pg = it < 32 ? __shfl_sync(0xffffffffu, my_page, it) : __ldcg(pt_u + (j >> 5));
        return (int)page_row(pg, j, p.pool_pages, p.status);
    }
    __device__ __forceinline__ void issue(const CUtensorMap& map, int row, int stage) const {             // lane 0
        const uint32_t bar = bars + stage * 8, dst = smem_addr(ring + stage * S::kTile);
        mbar_expect_tx(bar, S::kTile);
#pragma unroll
        for (int x = 0; x < S::kBoxes; ++x) tma_load_2d(dst + x * S::kBox, &map, x * (128 / Elem<T>::kBytes), row, bar);
    }
    // the appended token's row replaces whatever the copy fetched for its slot; rows past the unit's end become zero
    __device__ __forceinline__ void patch(unsigned char* tile, int j0, int n_valid, int which, int it) const {
        const int lane = threadIdx.x & 31;
        auto chunk_at = [&](int r, int c) { return tile + (c >> 3) * S::kBox + r * 128 + ((((c & 7) ^ r) & 7) << 4); };
        if (l_old >= j0 && l_old < j0 + kDcKeys) {
            const int row = row0(it);
            if (lane < S::kRow / 16) {
                const uint4 x = *reinterpret_cast<const uint4*>(newrow + which * S::kRow + lane * 16);
                *reinterpret_cast<uint4*>(chunk_at(l_old - j0, lane)) = x;
                unsigned char* storage = reinterpret_cast<unsigned char*>(which ? p.V : p.K);
                reinterpret_cast<uint4*>(storage + (size_t)(row + (l_old - j0)) * S::kRow)[lane] = x;
            }
            if (which == 0 && lane == 0) { p.word[(size_t)u * p.C + l_old] = 0u; p.pos[(size_t)u * p.C + l_old] = t; }
        }
        if (n_valid < kDcKeys)
            for (int x = lane; x < (kDcKeys - n_valid) * (S::kRow / 16); x += 32)
                *reinterpret_cast<uint4*>(chunk_at(n_valid + x / (S::kRow / 16), x % (S::kRow / 16))) = make_uint4(0, 0, 0, 0);
        __syncwarp();
    }
};

// The streaming loop in fp64 on the CUDA cores for NG heads: a key per lane, its channels shared by two half-warps; P.V by
// fp32 FMAs. qd: the queries as doubles [NG][D], pr: room for 16 x NG probabilities, lg: the block's logits [slot][NG].
// Magnitudes are whatever the inputs are: references and sums stay in fp64, a logit beyond fp32 is kept as an infinity (its
// verdict is formed again). push(h, m, Z): a head's sums go to the unit's blocks (the whole warp calls). A logit of +infinity makes its head's output NaN and no key important; so does NaN, but for bf16
// with 128 channels and up to four heads, where it counts for nothing: what the kernels for these shapes have always done
// (the block-per-split kernel there, the generic one elsewhere). Returns false if a wait expired.
template <typename T, int D, int GP, int NW, int NG, typename Push>
__device__ __forceinline__ bool dc_stream_fp64(const DcTiles<T, D, GP, NW>& c, const double* qd, float* pr, float* lg, float* rec, Push push) {
    using S = DcShape<T, D, GP>;
    constexpr int kKs = S::kKs, kVs = S::kVs, NC = D / 32;    // channels a lane accumulates
    constexpr int kHalf = S::kRow / 32, kEl = 16 / Elem<T>::kBytes;             // 16-byte chunks of half a row, elements of one
    // bf16: twice only, next to the tensor-core loop (a call costs that loop 2 %, all eight chunks unrolled 0.7 %, two nothing)
    constexpr int kUnroll = S::kBf16 ? 2 : kHalf;
    constexpr bool kNanPasses = !(S::kBf16 && D == 128 && GP <= 4);
    const int lane = threadIdx.x & 31, key = lane & 15, half = lane >> 4;
    bool failed = false, first = true;
    float acc[NG][NC];
    double Zl[NG], Mref[NG];
#pragma unroll
    for (int x = 0; x < NG; ++x) {
        Zl[x] = 0.0; Mref[x] = -INFINITY;
#pragma unroll
        for (int e = 0; e < NC; ++e) acc[x][e] = 0.f;
    }
    for (int it = 0; it < c.my_n; ++it) {
        const int j0 = c.first_key(it), n_valid = min(kDcKeys, c.k_end - j0);
        const int ks = it % kKs, vs = it % kVs;
        unsigned char* ktile = c.ring + ks * S::kTile;
        unsigned char* vtile = c.ring + (kKs + vs) * S::kTile;
        const bool edge = n_valid < kDcKeys || (c.l_old >= j0 && c.l_old < j0 + kDcKeys);
        if (!failed && !mbar_wait(c.bars + ks * 8, (it / kKs) & 1)) failed = true;
        if (edge) c.patch(ktile, j0, n_valid, 0, it);
        double s[NG];
#pragma unroll
        for (int x = 0; x < NG; ++x) s[x] = 0.0;
#pragma unroll kUnroll
        for (int i = 0; i < kHalf; ++i) {
            const int ch = half * kHalf + i;
            const uint4 raw = *reinterpret_cast<const uint4*>(ktile + (ch >> 3) * S::kBox + key * 128 + (((ch ^ key) & 7) << 4));
            double kd[kEl];
            if constexpr (S::kBf16) {
                unpack8_to_double(raw, kd);
            } else {
                kd[0] = (double)__uint_as_float(raw.x); kd[1] = (double)__uint_as_float(raw.y);
                kd[2] = (double)__uint_as_float(raw.z); kd[3] = (double)__uint_as_float(raw.w);
            }
#pragma unroll
            for (int x = 0; x < NG; ++x)
#pragma unroll
                for (int e = 0; e < kEl; e += 2) {
                    const double2 q = *reinterpret_cast<const double2*>(qd + x * D + ch * kEl + e);
                    s[x] = fma(q.x, kd[e], s[x]); s[x] = fma(q.y, kd[e + 1], s[x]);
                }
        }
        __syncwarp();
        if (it + kKs < c.my_n) {
            const int r0 = c.row0(it + kKs);
            if (lane == 0) { fence_async_smem(); c.issue(c.kmap, r0, ks); }
        }
        const bool on = key < n_valid;
        bool over = first;
#pragma unroll
        for (int x = 0; x < NG; ++x) {
            s[x] = (s[x] + __shfl_xor_sync(0xffffffffu, s[x], 16)) * inv_root_dim(D);
            over |= on && s[x] > Mref[x] + 16.0;
        }
        if (__any_sync(0xffffffffu, over)) {
#pragma unroll
            for (int x = 0; x < NG; ++x) {
                const double mn = fmax(Mref[x], warp_max(on && s[x] == s[x] ? s[x] : -INFINITY));
                const double sc = first || mn == -INFINITY ? 0.0 : exp_nonpos(Mref[x] - mn);
                Zl[x] *= sc;
                Mref[x] = mn;
#pragma unroll
                for (int e = 0; e < NC; ++e) acc[x][e] *= (float)sc;
            }
            first = false;
        }
#pragma unroll
        for (int x = 0; x < NG; ++x) {
            if (NG > 1 && (x & 1) != half) continue;          // the half-warps share the heads
            double ex = on ? exp_nonpos(s[x] - Mref[x]) : 0.0;
            if (on && (s[x] == INFINITY || (kNanPasses && s[x] != s[x]))) ex = NAN;
            if (NG > 1 || half == 0) {
                Zl[x] += ex;
                pr[key * NG + x] = (float)ex;
                if (on) lg[(j0 - c.k_begin + key) * NG + x] = s[x] == s[x] ? (float)s[x] : -INFINITY;
            }
        }
        __syncwarp();
        if (!failed && !mbar_wait(c.bars + (kKs + vs) * 8, (it / kVs) & 1)) failed = true;
        if (edge) c.patch(vtile, j0, n_valid, 1, it);
#pragma unroll 4
        for (int r = 0; r < kDcKeys; ++r) {
            const int at = lane * NC * Elem<T>::kBytes, ch = at >> 4;           // the lane's channels
            const unsigned char* src = vtile + (ch >> 3) * S::kBox + r * 128 + (((ch ^ r) & 7) << 4) + (at & 15);
            float v[NC];
            load_slice<T, NC>(reinterpret_cast<const T*>(src), v);
#pragma unroll
            for (int x = 0; x < NG; ++x) {
                const float pj = pr[r * NG + x];
#pragma unroll
                for (int e = 0; e < NC; ++e) acc[x][e] = fmaf(pj, v[e], acc[x][e]);
            }
        }
        __syncwarp();
        if (it + kVs < c.my_n) {
            const int r0 = c.row0(it + kVs);
            if (lane == 0) { fence_async_smem(); c.issue(c.vmap, r0, kKs + vs); }
        }
    }
#pragma unroll
    for (int x = 0; x < NG; ++x) {
        Zl[x] = warp_sum(Zl[x]);
        push(x, Mref[x], Zl[x]);
#pragma unroll
        for (int e = 0; e < NC; ++e) rec[x * D + lane * NC + e] = acc[x][e];
    }
    return !failed;
}

template <typename T, int D, int GP, int NW>
__global__ void __launch_bounds__(NW * 32, dc_blocks<T, D, GP, NW>())
decode_cluster_kernel(const __grid_constant__ DecodeClusterParams dp, const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap) {
    extern __shared__ __align__(1024) unsigned char smem[];
    using S = DcShape<T, D, GP>;
    constexpr bool kBf16 = S::kBf16;
    constexpr int NT = NW * 32, kKs = S::kKs, kVs = S::kVs, kMaxWords = dc_max_words<T, D, GP, NW>();
    static_assert(dc_ring_holds_lists<T, D, GP, NW>(), "keep bits, lists and prefix sums lie in the ring");
    constexpr int NH = kBf16 ? (GP == 8 ? 2 : 1) : GP;        // heads a thread handles logits of
    constexpr int NK = kBf16 ? 2 : 1;                         // keys of a tile a thread handles
    const DecodeParams& p = dp.p;
    const int G = kBf16 && GP == 2 ? dp.G : GP;               // one or two heads share an instance
    const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cs0 = (int)cluster_size(), rank0 = (int)cluster_rank();            // (read again behind the loop, which has no registers to spare)
    const DcSmem lay = dc_smem_layout<T, D, GP, NW>(0);       // the logits come last: every other offset is a constant
    unsigned char* ring = smem + warp * S::kWarpRing;
    unsigned char* prob = smem + lay.prob + warp * S::kProb;
    unsigned char* newrow = smem + lay.newrow;
    const uint32_t bars = smem_addr(smem + lay.bars) + warp * S::kStages * 8;
    DcMisc<NW, GP>* misc = reinterpret_cast<DcMisc<NW, GP>*>(smem + lay.misc);
    const uint32_t xbar = smem_addr(misc->bar);

    // ---- set-up that reads nothing of the previous launch ----
    if (tid == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&kmap)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&vmap)) : "memory");
        misc->n_open = 0;
#pragma unroll
        for (int x = 0; x < NW; ++x) misc->flags[x] = 0u;
#pragma unroll
        for (int x = 0; x < kDcBars; ++x) mbar_init(xbar + x * 8, x < kDcMeet ? 1 : cs0);
    }
    if (lane == 0) {
#pragma unroll
        for (int s = 0; s < S::kStages; ++s) mbar_init(bars + s * 8, 1);
        fence_mbar_init();
        fence_async_smem();
    }
    cluster_arrive();                                         // the barriers are there before anybody's first push (cluster_wait below)
    int l_old;
    uint32_t state = smem_addr(smem) & 1023u ? kDcExpired : 0u;          // swizzled tiles need the alignment; never expected
    if (p.chain_wait) {                                       // this unit's previous step, not the whole previous launch
        if (p.early_trigger) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        if (tid == 0) misc->stamp = wait_unit_stamp(p.unit_stamp + u, (uint32_t)p.step, p.status);
        __syncthreads();
        const unsigned long long sw = misc->stamp;
        const bool ok = (uint32_t)(sw >> 32) == (uint32_t)p.step;
        l_old = ok ? (int)(uint32_t)sw : 0;
        if (!ok) state = kDcExpired;
        asm volatile("fence.proxy.async.global;" ::: "memory");   // the tile copies read rows that ordinary stores wrote
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        l_old = __ldcg(p.live_in + u);
    }
    // queries, and in the block that will own the last slot the appended rows: requested next to the length (their latency
    // is a bus round trip when the caller's buffers are host memory)
    const float* q_raw = reinterpret_cast<const float*>(p.q) + (size_t)u * G * D;
    if constexpr (kBf16)
        for (int x = tid; x < G * (S::kRow / 16); x += NT)
            cp_async16(smem_addr(smem + lay.q + x * 16), reinterpret_cast<const unsigned char*>(p.q) + ((size_t)u * G * (S::kRow / 16) + x) * 16);
    if (rank0 == cs0 - 1)
        for (int x = tid; x < 2 * (S::kRow / 16); x += NT) {
            const int c = x % (S::kRow / 16);
            cp_async16(smem_addr(newrow + x * 16), reinterpret_cast<const unsigned char*>(x < S::kRow / 16 ? p.k_new : p.v_new) + (size_t)u * S::kRow + c * 16);
        }
    const uint32_t kmax_old = kBf16 ? __ldcg(p.kmax + u) : 0u;
    const int32_t* pt_u = p.page_table ? p.page_table + (size_t)u * p.pt_stride : nullptr;
    const int room = pt_u ? __ldcg(p.page_room + u) : 1;
    const int b = u / p.Hkv;
    const int t = __ldcg(p.base_tokens + b) + p.step + 1;
    const bool evict_on = min(p.w, __ldcg(p.base_obs + b) + p.step + 1) >= p.w;
    if (p.early_trigger && !p.chain_wait) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the block has its length
    const int l = l_old + 1;
    if (l > p.C || !room) state |= kDcFull;
    if (tid == NT - 1) misc->log_t = log((double)t);
    // the block's slots: whole words, shared out evenly
    const int n_words = state ? 0 : (l + 31) >> 5;
    auto word_begin = [&](int o, int cs) -> int { return (int)((uint32_t)(n_words * o) / (uint32_t)cs); };
    const int w0 = word_begin(rank0, cs0), w1 = word_begin(rank0 + 1, cs0);
    // the outputs are shared out over the blocks, two channels at a time
    constexpr int kHalfD = D / 2;
    auto first_pair = [&](int o, int cs) { return G * kHalfD * o / cs; };
    if (tid == 0) {                                           // what will be pushed into this block
        mbar_expect_tx(xbar + kDcRecords * 8, cs0 * NW * (G * 16 + 4));
        mbar_expect_tx(xbar + kDcOutputs * 8, cs0 * (first_pair(rank0 + 1, cs0) - first_pair(rank0, cs0)) * 8);
        mbar_expect_tx(xbar + kDcCounts * 8, cs0 * NW * 8 + min(32, n_words) * (4 + 128) + (rank0 < cs0 - 1 ? 2 * S::kRow : 0));
    }
    const int k_begin = w0 * 32, k_end = state ? 0 : min(l, w1 * 32), n_keys = max(0, k_end - k_begin);
    const int n_tiles = (n_keys + kDcKeys - 1) / kDcKeys;
    const int my_n = n_tiles > warp ? (n_tiles - warp + NW - 1) / NW : 0;       // tiles warp, warp + NW, ...
    const bool fits = n_keys * G <= dp.lcap;
    float* lg = fits ? reinterpret_cast<float*>(smem + lay.logits)
                     : reinterpret_cast<float*>(p.stash + (size_t)u * G * p.C) + (size_t)k_begin * G;   // the unit's own scratch: launches overlap
    int my_page = 0;
    if (pt_u) {
        const int j = k_begin + (warp + lane * NW) * kDcKeys;
        if (j < k_end) my_page = __ldcg(pt_u + (j >> 5));
    }
    const DcTiles<T, D, GP, NW> tiles{p, kmap, vmap, pt_u, ring, newrow, bars, u, l_old, t, k_begin, k_end, my_n, my_page};
#pragma unroll
    for (int it = 0; it < (kKs > kVs ? kKs : kVs); ++it)
        if (it < my_n) {
            const int r0 = tiles.row0(it);
            if (lane == 0) { if (it < kKs) tiles.issue(kmap, r0, it); if (it < kVs) tiles.issue(vmap, r0, kKs + it); }
        }
    cp_async_wait_all();
    if (!kBf16) {
        double* qd = reinterpret_cast<double*>(smem + lay.q);
        for (int x = tid; x < G * D; x += NT) qd[x] = q_raw[x];
    }
    __syncthreads();
    cluster_wait();

    // ---- 1. streaming ----
    const double inv_root_d = inv_root_dim(D);
    uint32_t* wordu = p.word + (size_t)u * p.C;
    int32_t* posu = p.pos + (size_t)u * p.C;
    bool failed = false;
    float* rec = reinterpret_cast<float*>(ring);              // the warp's record [G][D], once its tiles are done
    auto push_sums = [&](int h, double m, double z, int peer) {                // a head's {m, Z} of this warp, to one block
        const uint32_t at = smem_addr(&misc->rec[h][cluster_rank() * NW + warp]);
        push_2f64(map_rank(at, peer), m, z, map_rank(xbar + kDcRecords * 8, peer));
    };
    auto push_all = [&](int h, double m, double z) { if (lane < (int)cluster_size()) push_sums(h, m, z, lane); };

    if constexpr (kBf16) {
        // pieces of the queries, as B fragments (column n = lane / 4): every warp needs all of them, so a warp cuts the
        // queries' channels 16 kk.. of kk = warp, warp + NW, ... and the others read them from shared memory
        constexpr int KK = D / 16, kPieces = S::kPieces;
        uint32_t* pieces = reinterpret_cast<uint32_t*>(smem + lay.pieces);      // [KK][kPieces / 2][32 lanes][2]
        uint32_t qmax = 0u;                                   // largest magnitude of the unit's queries, as kmax
        auto too_wide = [&](uint32_t k) {                     // of keys of up to this magnitude
            const float reach = __uint_as_float(k << 16) * __uint_as_float(qmax << 16);
            return max(k, qmax) >= kSplitMaxBits || reach > kDcReach || reach * (float)l > dc_reach_keys<GP>(G);
        };
        {
            const int n = lane >> 2;
            const int hq = GP == 8 ? n : GP == 4 ? n >> 1 : (n & 3) >> 1;
            const bool on = hq < G;
            const uint32_t* src = reinterpret_cast<const uint32_t*>(smem + lay.q) + (on ? hq : 0) * (D / 2) + (lane & 3);
            uint32_t mx = 0u;
#pragma unroll
            for (int kk = 0; kk < KK; ++kk) mx = max_abs_bf16x2(max_abs_bf16x2(mx, src[kk * 8]), src[kk * 8 + 4]);
            uint32_t m16 = on ? max(mx & 0xffffu, mx >> 16) : 0u;
            m16 = max(m16, __shfl_xor_sync(0xffffffffu, m16, 1));
            m16 = max(m16, __shfl_xor_sync(0xffffffffu, m16, 2));
            const bool ok = m16 < kSplitMaxBits;
            qmax = __reduce_max_sync(0xffffffffu, m16);
            if (too_wide(kmax_old)) state |= kDcWide;
            if (tid == 0) misc->cut_for = state & kDcWide ? 0u : kmax_old;
            const float c = split_query_const(ok ? __uint_as_float(m16 << 16) : 1.f);
            float n1 = 0.f, n2 = 0.f, n3 = 0.f;
            for (int kk = warp; kk < KK; kk += NW) {
                uint32_t w[kPieces];
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const uint32_t raw = on ? src[kk * 8 + hf * 4] : 0u;
                    const float a[2] = {__uint_as_float(raw << 16), __uint_as_float(raw & 0xffff0000u)};
                    uint32_t y1[2], y2[2], y3[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float x1, x2, x3;
                        split_query(a[e], c, x1, x2, x3);
                        n1 += fabsf(a[e]); n2 += fabsf(x2); n3 += fabsf(x3);
                        y1[e] = __float_as_uint(x1); y2[e] = __float_as_uint(x2); y3[e] = __float_as_uint(x3);
                    }
                    auto pack = [](const uint32_t (&y)[2]) { return (y[0] >> 16) | (y[1] & 0xffff0000u); };   // exact: bf16 numbers
                    if constexpr (GP == 8) {
                        w[hf] = pack(y1); w[2 + hf] = pack(y2); w[4 + hf] = pack(y3);
                    } else if constexpr (GP == 4) {
                        w[hf] = n & 1 ? pack(y2) : pack(y1);
                        w[2 + hf] = n & 1 ? 0u : pack(y3);
                    } else {
                        w[hf] = n & 4 ? (n & 1 ? 0u : pack(y3)) : n & 1 ? pack(y2) : pack(y1);
                    }
                }
#pragma unroll
                for (int x = 0; x < kPieces; x += 2)
                    *reinterpret_cast<uint2*>(pieces + ((kk * (kPieces / 2) + x / 2) * 32 + lane) * 2) = make_uint2(w[x], w[x + 1]);
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                n1 += __shfl_xor_sync(0xffffffffu, n1, o);
                n2 += __shfl_xor_sync(0xffffffffu, n2, o);
                n3 += __shfl_xor_sync(0xffffffffu, n3, o);
            }
            // Error of a logit (before the 1/sqrt(d)) per unit of the unit's largest key magnitude A, this warp's channels'
            // share. r2.q: per 16 channels 17 roundings of 2^-23 (a product of 16 terms and its accumulator; twice that for
            // eight heads, whose two products share one) and 8 of 2^-24 in fp32, on terms of at most A/8192 |q|; k.q3: at
            // most 2 * 8 * 17 roundings of 2^-23; r2.q3 <= A/8192 |q3| (left out for eight and four heads); the sum of the
            // small parts (k2.q2 <= A/64 |q2| among them) rounds three times.
            if (on && (lane & 3) == 0)
                misc->qe_part[warp][hq] = dp.bound_scale * 1.05f * ((GP == 8 ? 4.6e-6f : 2.6e-6f) * (n1 * 1.01f) * (1.f / 8192.f) + (3.3e-5f + 1.3e-4f) * n3 + 2.4e-7f * n2 * (1.f / 64.f));
        }
        __syncthreads();
        // The keys are cut on a grid of the unit's, kept in p.kmax: the largest magnitude it has ever held (scanning every
        // tile for its own cost 96 instructions of 550 per tile and a chain of 32 dependent ones).
        uint32_t kmax = kmax_old;
        if (cluster_rank() == cluster_size() - 1) {
            uint32_t m = 0u;
            if (lane < S::kRow / 16) {
                const uint4 x = *reinterpret_cast<const uint4*>(newrow + lane * 16);
                m = max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(m, x.x), x.y), x.z), x.w);
            }
            kmax = max(kmax, __reduce_max_sync(0xffffffffu, max(m & 0xffffu, m >> 16)));
        }
        if (too_wide(kmax)) state |= kDcWide;
        if (tid < G) {
            float e = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w) e += misc->qe_part[w][tid];
            misc->qe[tid] = e * 1.0001f;
        }
        if (state & kDcWide) {
            double* qd = reinterpret_cast<double*>(pieces);
            for (int x = tid; x < G * D; x += NT) qd[x] = (double)Elem<bf16_t>::load(reinterpret_cast<const bf16_t*>(smem + lay.q) + x);
            __syncthreads();
            float* pr = reinterpret_cast<float*>(prob);
            if constexpr (GP == 2) {
                if (G == 1) failed = !dc_stream_fp64<T, D, GP, NW, 1>(tiles, qd, pr, lg, rec, push_all);
                else failed = !dc_stream_fp64<T, D, GP, NW, 2>(tiles, qd, pr, lg, rec, push_all);
            } else {
                failed = !dc_stream_fp64<T, D, GP, NW, GP>(tiles, qd, pr, lg, rec, push_all);
            }
        } else {
            uint32_t b1[KK][2], b2[GP == 2 ? 1 : KK][2], b3[GP == 8 ? KK : 1][2];
#pragma unroll
            for (int kk = 0; kk < KK; ++kk) {
                const uint2* src = reinterpret_cast<const uint2*>(pieces) + kk * (kPieces / 2) * 32 + lane;
                const uint2 x = src[0];
                b1[kk][0] = x.x; b1[kk][1] = x.y;
                if constexpr (kPieces > 2) { const uint2 y = src[32]; b2[kk][0] = y.x; b2[kk][1] = y.y; }
                if constexpr (kPieces > 4) { const uint2 z = src[64]; b3[kk][0] = z.x; b3[kk][1] = z.y; }
            }
            double Zl[NH];
            float Mref[NH];
#pragma unroll
            for (int x = 0; x < NH; ++x) { Zl[x] = 0.0; Mref[x] = -INFINITY; }
            float accd[D / 16][4];
#pragma unroll
            for (int cb = 0; cb < D / 16; ++cb)
#pragma unroll
                for (int e = 0; e < 4; ++e) accd[cb][e] = 0.f;
            const SplitGrid g = split_grid(kmax);
            const int h0 = GP == 8 ? 2 * (lane & 3) : (lane & 3);                    // the thread's head(s)
            // Lane offsets of the fragment loads inside a tile. Rows are 128 bytes and a tile starts on a multiple of 1024, so
            // 16-byte chunk c of the lane's row (at c ^ row mod 8) is one exclusive-or away from chunk 0 or 1.
            const uint32_t klane = (lane & 15) * 128 + (((lane >> 4) ^ (lane & 7)) << 4);
            const uint32_t vlane = (((lane >> 4) << 3) + (lane & 7)) * 128 + ((((lane >> 3) & 1) ^ (lane & 7)) << 4);
            const uint32_t ring_a = smem_addr(ring);
            bool first = true;
            // The tile that needs patching (keys past the block's end, or the appended slot, which is the unit's last) is the
            // block's last one.
            const int whole = k_end == l ? n_keys - 1 : n_keys;
            float* lgp = lg + (warp * kDcKeys + (lane >> 2)) * G + h0;
            int left = n_keys - warp * kDcKeys;                   // keys from the tile's first on
            for (int it = 0; it < my_n; ++it, left -= NW * kDcKeys, lgp += NW * kDcKeys * G) {
                const int n_valid = min(kDcKeys, left);
                const int ks = it % kKs, vs = it % kVs;
                const bool edge = n_keys - left + kDcKeys > whole;
                if (!failed && !mbar_wait(bars + ks * 8, (it / kKs) & 1)) failed = true;   // once one wait has expired the rest are skipped
                if (edge) tiles.patch(ring + ks * S::kTile, k_end - left, n_valid, 0, it);
                const uint32_t arow = ring_a + ks * S::kTile + klane;
                uint32_t a[4][4];                                 // 64 channels of the tile at a time
                // sums of the products of pieces; see the head of the file
                float x1[4], x2[4], x3[4], x4[4], lo[4];
#pragma unroll
                for (int kk = 0; kk < KK; ++kk) {
                    if (kk % 4 == 0) {
#pragma unroll
                        for (int x = 0; x < 4; ++x) ldmatrix_x4(a[x], (arow ^ (x << 5)) + (kk >> 2) * S::kBox);
                        if (kk + 4 == KK) {                       // the rest of the tile is in registers: its stage is free
                            __syncwarp();
                            if (it + kKs < my_n) {
                                const int r0 = tiles.row0(it + kKs);
                                if (lane == 0) tiles.issue(kmap, r0, ks);
                            }
                        }
                    }
                    uint32_t k1[4], k2[4], r2[4];
                    split_key(a[kk % 4], g, k1, k2, r2);
                    float tt[4];
                    auto mma = [&](float (&d)[4], const uint32_t (&x)[4], const uint32_t (&b)[2]) {   // the sum's first term, or one more
                        if (kk == 0) mma16816_zero(d, x, b[0], b[1]); else mma16816(d, x, b[0], b[1]);
                    };
                    mma(x1, k1, b1[kk]);
                    mma16816_zero(tt, r2, b1[kk][0], b1[kk][1]);
                    if constexpr (GP == 8) {
                        mma(x2, k1, b2[kk]);                      // k1.q2 + k2.q1: exact together
                        mma16816(x2, k2, b1[kk][0], b1[kk][1]);
                        mma(x4, k2, b2[kk]);                      // exact
                        mma16816(tt, r2, b2[kk][0], b2[kk][1]);
                        mma(x3, k1, b3[kk]);
                        mma16816(x3, k2, b3[kk][0], b3[kk][1]);
                    } else {
                        mma(x2, k2, b1[kk]);
                        if constexpr (GP == 4) {
                            mma(x3, k1, b2[kk]);
                            mma(x4, k2, b2[kk]);
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) lo[e] = kk == 0 ? tt[e] : lo[e] + tt[e];
                }
                // Eq. 2's exponent, thread's keys lane / 4 and + 8
                double s[NK][NH];
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    if constexpr (GP == 8) {
#pragma unroll
                        for (int x = 0; x < 2; ++x) {
                            const int e = 2 * y + x;
                            s[y][x] = (((double)x1[e] + (double)x2[e]) + (double)(x4[e] + (lo[e] + x3[e]))) * inv_root_d;
                        }
                    } else {
                        // columns: (.q1, .q2) of the thread's head; two heads: the q3 products two lanes further on
                        float small = x2[2 * y + 1] + (lo[2 * y] + lo[2 * y + 1]);
                        if constexpr (GP == 4) small += x3[2 * y] + x4[2 * y];
                        else small += __shfl_xor_sync(0xffffffffu, x1[2 * y] + (x2[2 * y] + lo[2 * y]), 2);
                        s[y][0] = (((double)x1[2 * y] + (double)(x1[2 * y + 1] + x2[2 * y])) + (double)small) * inv_root_d;
                    }
                }
                bool on[NK][NH];
                bool over = first;
#pragma unroll
                for (int y = 0; y < 2; ++y)
#pragma unroll
                    for (int x = 0; x < NH; ++x) {
                        on[y][x] = (lane >> 2) + 8 * y < n_valid && h0 + x < G;
                        over |= on[y][x] && (float)s[y][x] > Mref[x] + 16.f;
                    }
                if (__any_sync(0xffffffffu, over)) {              // the reference moves: first tile, or a logit far above it (rare)
                    float scf[NH];
#pragma unroll
                    for (int x = 0; x < NH; ++x) {
                        float mt = fmaxf(on[0][x] ? (float)s[0][x] : -INFINITY, on[1][x] ? (float)s[1][x] : -INFINITY);
#pragma unroll
                        for (int o = 4; o < 32; o <<= 1) mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, o));
                        const float mn = fmaxf(Mref[x], mt);
                        const double sc = first || mn == -INFINITY ? 0.0 : exp_nonpos((double)Mref[x] - (double)mn);
                        Zl[x] *= sc;
                        scf[x] = (float)sc;
                        Mref[x] = mn;
                    }
                    if constexpr (GP == 2) {                      // lanes 2 and 3 of four accumulate the third parts of heads 0 and 1
                        const float o = __shfl_xor_sync(0xffffffffu, scf[0], 2);
                        if (lane & 2) scf[0] = o;
                    }
#pragma unroll
                    for (int cb = 0; cb < D / 16; ++cb)           // the accumulators' columns are the thread's own heads
#pragma unroll
                        for (int e = 0; e < 4; ++e) accd[cb][e] *= GP == 8 ? scf[(e & 1) % NH] : scf[0];
                    first = false;
                }
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    const int kq = (lane >> 2) + 8 * y;
                    float pf[NH];
#pragma unroll
                    for (int x = 0; x < NH; ++x) {
                        const float sf = (float)s[y][x];
                        const double ex = exp_nonpos_where(on[y][x] && sf - Mref[x] > -700.f, s[y][x] - (double)Mref[x]);
                        Zl[x] += ex;
                        pf[x] = (float)ex;
                        if (on[y][x]) lgp[8 * y * G + x] = sf;
                    }
                    uint32_t* const dst = reinterpret_cast<uint32_t*>(prob + kq * 16) + (lane & 3);
                    if constexpr (GP == 8) {                      // [key][8 heads] first parts, then second, then third
#pragma unroll
                        for (int part = 0; part < 3; ++part) {
                            const uint32_t w = pack_bf16x2(pf[1 % NH], pf[0]);
                            dst[part * 64] = w;
                            pf[0] -= __uint_as_float(w << 16);
                            pf[1 % NH] -= __uint_as_float(w & 0xffff0000u);
                        }
                    } else {                                      // [key][head x (first, second)], and (third, 0) behind them
                        const uint32_t a = pack_bf16x2(0.f, pf[0]) << 16;
                        const float r = pf[0] - __uint_as_float(a);
                        const uint32_t b = pack_bf16x2(r, 0.f) & 0xffff0000u, c = pack_bf16x2(0.f, r - __uint_as_float(b));
                        if constexpr (GP == 4) {
                            dst[0] = b | (a >> 16);
                            dst[64] = c;
                        } else if (h0 < 2) {
                            dst[0] = b | (a >> 16);
                            dst[2] = c;
                        }
                    }
                }
                __syncwarp();
                if (!failed && !mbar_wait(bars + (kKs + vs) * 8, (it / kVs) & 1)) failed = true;
                if (edge) tiles.patch(ring + (kKs + vs) * S::kTile, k_end - left, n_valid, 1, it);
                {
                    uint32_t bf[4];
                    ldmatrix_x4_trans(bf, smem_addr(prob) + (GP > 2 ? lane : lane & 15) * 16);        // keys 0-7 | 8-15 (| the next parts)
                    uint32_t b3p[2];
                    if constexpr (GP == 8) ldmatrix_x2_trans(b3p, smem_addr(prob) + 512 + (lane & 15) * 16);
                    const uint32_t vrow = ring_a + (kKs + vs) * S::kTile + vlane;
#pragma unroll
                    for (int cb = 0; cb < D / 16; ++cb) {
                        uint32_t va[4];
                        ldmatrix_x4_trans(va, (vrow ^ ((cb & 3) << 5)) + (cb >> 2) * S::kBox);
                        mma16816(accd[cb], va, bf[0], bf[1]);     // Eq. 1
                        if constexpr (GP > 2) mma16816(accd[cb], va, bf[2], bf[3]);
                        if constexpr (GP == 8) mma16816(accd[cb], va, b3p[0], b3p[1]);
                    }
                }
                __syncwarp();
                if (it + kVs < my_n) {
                    const int r0 = tiles.row0(it + kVs);
                    if (lane == 0) tiles.issue(vmap, r0, kKs + vs);
                }
            }
#pragma unroll
            for (int x = 0; x < NH; ++x) {
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) Zl[x] += __shfl_xor_sync(0xffffffffu, Zl[x], o);
                if ((lane >> 2) < (int)cluster_size() && h0 + x < G) push_sums(h0 + x, (double)Mref[x], Zl[x], lane >> 2);
            }
#pragma unroll
            for (int cb = 0; cb < D / 16; ++cb) {
                if constexpr (GP == 8) {
                    rec[h0 * D + cb * 16 + (lane >> 2)] = accd[cb][0];
                    rec[(h0 + 1) * D + cb * 16 + (lane >> 2)] = accd[cb][1];
                    rec[h0 * D + cb * 16 + 8 + (lane >> 2)] = accd[cb][2];
                    rec[(h0 + 1) * D + cb * 16 + 8 + (lane >> 2)] = accd[cb][3];
                } else {
                    float a0 = accd[cb][0] + accd[cb][1], a1 = accd[cb][2] + accd[cb][3];  // the parts' sums
                    if constexpr (GP == 2) {
                        a0 += __shfl_xor_sync(0xffffffffu, a0, 2);
                        a1 += __shfl_xor_sync(0xffffffffu, a1, 2);
                    }
                    if (h0 < G) {
                        rec[h0 * D + cb * 16 + (lane >> 2)] = a0;
                        rec[h0 * D + cb * 16 + 8 + (lane >> 2)] = a1;
                    }
                }
            }
        }
        state = (state & ~0xffffu) | kmax;
    } else {
        failed = !dc_stream_fp64<T, D, GP, NW, GP>(tiles, reinterpret_cast<const double*>(smem + lay.q), reinterpret_cast<float*>(prob), lg, rec, push_all);
        if (warp == 0 && lane < GP) misc->qe[lane] = 0.f;
    }
    const int cs = (int)cluster_size(), rank = (int)cluster_rank();
    if (failed) state |= kDcExpired;
    state = __reduce_or_sync(0xffffffffu, state);             // the magnitude is the same in every lane
    if (lane == 0 && (state & kDcExpired)) report_status(p.status, CORM_ERR_TIMEOUT);
    if (lane < cs) push_u32(map_rank(smem_addr(&misc->state[rank * NW + warp]), lane), state, map_rank(xbar + kDcRecords * 8, lane));
    // the next launch may become resident while this one judges and compacts (it waits for this one to complete)
    if (!p.early_trigger) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // registers and positions of the first slots this thread judges are requested before the blocks meet
    constexpr int kB = GP == 8 ? 4 : 8;                       // slots per thread and batch
    uint32_t wv[kB];
    int32_t pv[kB];
    float sv[kB][GP];
    auto load_regs = [&](int base) {
#pragma unroll
        for (int k = 0; k < kB; ++k) {
            const int i = base + k * NT + tid, j = k_begin + i;
            wv[k] = 0u; pv[k] = t;                            // the token appended by this step
            if (i - lane >= n_keys) continue;
            if (j < k_end && j < l_old) { wv[k] = __ldcg(wordu + j); pv[k] = __ldcg(posu + j); }
        }
        // (two branches: the addresses' space has to be known for one wide load per slot)
        if (fits) {
            const float* ls = reinterpret_cast<const float*>(smem + lay.logits);
#pragma unroll
            for (int k = 0; k < kB; ++k)
                if (base + k * NT + tid < n_keys) load_logits<GP, false>(ls + (base + k * NT + tid) * G, G, sv[k]);
        } else {
#pragma unroll
            for (int k = 0; k < kB; ++k)
                if (base + k * NT + tid < n_keys) load_logits<GP, true>(lg + (size_t)(base + k * NT + tid) * G, G, sv[k]);
        }
    };
    __syncthreads();                                          // the appended slot's row, word and position are stored
    load_regs(0);
    bool late = !mbar_wait_cluster(xbar + kDcRecords * 8, 0);                   // a push that should have been here
    // A block that misses pushes stays until its peers are done: the cluster's barrier counts blocks that have ended as there.
    auto leave = [&](bool full) {
        if (late) report_status(p.status, CORM_ERR_TIMEOUT);
        if (rank == 0 && tid == 0) {                          // the unit is left as it is
            if (full) report_status(p.status, CORM_ERR_CAPACITY);
            p.live_out[u] = l_old;
            if (full) publish_unit_stamp(p, u, l_old);
            report_live(p, u, p.step + 1, l_old);
        }
        if (late) cluster_sync();
    };

    // ---- thresholds of Definition 3.1 in log form, the same in every block: warp h reduces head h over the unit's warps ----
    constexpr int kEnt = kDcMaxCluster * NW / 32;             // (block, warp) entries per lane
    uint32_t unit_state = 0u;
#pragma unroll
    for (int y = 0; y < kEnt; ++y)
        if (y * 32 + lane < cs * NW) unit_state = max(unit_state, misc->state[y * 32 + lane]);
    unit_state = __reduce_max_sync(0xffffffffu, unit_state);
    late = __syncthreads_or(late);
    if (late) unit_state |= kDcExpired;
    if (unit_state & (kDcExpired | kDcFull)) {
        leave(!(unit_state & kDcExpired) || l > p.C || !room);
        return;
    }
    // the appended key enters the unit's magnitude whatever became of the queries (every block has read the old one)
    if (kBf16 && rank == 0 && tid == 0) p.kmax[u] = unit_state & 0xffffu;
    // error of a head's log-sum-exp per unit of qe (every logit of it is off by at most this much): from the magnitude the
    // keys were cut for. Where the appended key sent its block to the fp64 loop the others cut for the one before it.
    const uint32_t cut_for = unit_state & kDcWide ? misc->cut_for : unit_state & 0xffffu;
    const float eps_a = kBf16 && (cut_for || !(unit_state & kDcWide)) ? split_amax(cut_for) * (float)inv_root_d * 1.0001f : 0.f;
    // The appended row goes to the blocks, one of which may move it into a hole: by the warps that have no head here.
    if (rank == cs - 1 && (G >= NW || warp >= G)) {
        constexpr int kNew = 2 * S::kRow / 16;
        const int first = G >= NW ? 0 : G * 32;
        for (int x = tid - first; x < (cs - 1) * kNew; x += NT - first)
            push_v4(map_rank(smem_addr(newrow + x % kNew * 16), x / kNew), *reinterpret_cast<const uint4*>(newrow + x % kNew * 16),
                    map_rank(xbar + kDcCounts * 8, x / kNew));
    }
    for (int h = warp; h < G; h += NW) {
        double m[kEnt], z[kEnt], M = -INFINITY, Z = 0.0;
#pragma unroll
        for (int y = 0; y < kEnt; ++y) {
            const bool on = y * 32 + lane < cs * NW;
            m[y] = on ? misc->rec[h][y * 32 + lane].m : -INFINITY;
            z[y] = on ? misc->rec[h][y * 32 + lane].z : 0.0;
            M = fmax(M, m[y]);
        }
        M = warp_max(M);
#pragma unroll
        for (int y = 0; y < kEnt; ++y) {
            const double sc = m[y] == -INFINITY ? 0.0 : exp_nonpos(m[y] - M);
            Z = fma(z[y], sc, Z);
            if ((y * 32 + lane) / NW == rank) misc->sc[h][(y * 32 + lane) % NW] = (float)sc;
        }
        Z = warp_sum(Z);                                      // a fixed tree: every block gets the same bits
        if (lane == 0) {
            const double thr = M + log(Z) + p.log_alpha - misc->log_t;
            const float tf = thr == thr ? (float)thr : INFINITY, ta = fabsf(tf);     // behind a NaN no key is important
            misc->thr[h] = thr; misc->Zt[h] = Z; misc->thr_f[h] = tf;
            misc->slack[h] = (eps_a > 0.f ? 2.f * eps_a * misc->qe[h] : 0.f) + (ta < 3e38f ? ta : 0.f) * 1.3e-7f + 1e-12f;
        }
    }
    __syncthreads();

    // ---- 2. verdicts, register update, keep bits ----
    uint32_t* keep = reinterpret_cast<uint32_t*>(smem + kDcRecBytes);           // the ring is free behind the warps' records
    // Pushes don't order a block's ordinary stores for the others, so what a row move needs of this step, the registers of the
    // unit's last 32 words and the appended row, is pushed too. us per request with a release (an arrival on a barrier of its own)
    // instead / with these pushes: tiny fp32 721 / 682, 32 layers 11004 / 10705, G 8 1255 / 1223, 64 channels 1293 / 1232, fp32
    // 728 / 699, but G 4 5846 / 5880 and 6042 / 6137 (more registers than there are behind the loop of that instance).
    uint32_t* tail_regs = reinterpret_cast<uint32_t*>(smem + NW * S::kWarpRing - kDcRegBytes);
    const int tail_slot = (n_words - 32) * 32;                // the first of them (negative in short units)
    // the block's share of the unit's output numerators, as the blocks push it: [block][pair]
    const int np = G * kHalfD, pair0 = first_pair(rank, cs), pair1 = first_pair(rank + 1, cs), pair_cap = (np + cs - 1) / cs;
    float2* outputs = reinterpret_cast<float2*>(smem + (kBf16 ? lay.pieces : lay.q));           // (every warp is done with the queries)
    int n_imp = 0, n_keep = 0;
    {
        // first the numerators (Eq. 1) of the block's slots, its warps' records merged, each to the block that writes it
        const int shift = 31 - __clz(kHalfD) + __popc(G - 1);
        for (int x = tid; x < np; x += NT) {
            const int h = x / kHalfD;
            float a0 = 0.f, a1 = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const float sc = misc->sc[h][w];
                const float2 v = reinterpret_cast<const float2*>(smem + w * S::kWarpRing)[x];
                a0 += sc != 0.f ? v.x * sc : 0.f;
                a1 += sc != 0.f ? v.y * sc : 0.f;
            }
            const int owner = ((x + 1) * cs - 1) >> shift, first = first_pair(owner, cs);        // the last one with first <= x
            push_2u32(map_rank(smem_addr(outputs + rank * pair_cap + (x - first)), owner), __float_as_uint(a0), __float_as_uint(a1),
                      map_rank(xbar + kDcOutputs * 8, owner));
        }
        if (n_keys > (S::kWarpRing - kDcRecBytes) * 8) __syncthreads();          // so many keep bits reach the second warp's record
        float tf[GP], sl[GP];
#pragma unroll
        for (int h = 0; h < GP; ++h) { tf[h] = h < G ? misc->thr_f[h] : INFINITY; sl[h] = h < G ? misc->slack[h] : 0.f; }
#pragma unroll 1
        for (int base0 = 0; base0 < n_keys; base0 += kB * NT) {
            if (base0) load_regs(base0);
            uint32_t imp = 0u, open[kB];
#pragma unroll
            for (int k = 0; k < kB; ++k) {
                const int i = base0 + k * NT + tid;
                open[k] = 0u;
                if (i - lane >= n_keys) continue;             // uniform in the warp
                bool sure = false;
                uint32_t near = 0u;
#pragma unroll
                for (int h = 0; h < GP; ++h) {
                    const float sf = sv[k][h], margin = sf - tf[h], err = fmaf(fabsf(sf), 6.1e-8f, sl[h]);
                    sure |= margin >= err;
                    near |= !(margin <= -err) ? 1u << h : 0u; // (two infinities: to be formed again)
                }
                open[k] = i < n_keys && !sure ? near : 0u;
                imp |= i < n_keys && sure ? 1u << k : 0u;
            }
            uint32_t any_open = 0u;
#pragma unroll
            for (int k = 0; k < kB; ++k) any_open |= open[k];
            if (__any_sync(0xffffffffu, any_open != 0u)) {    // rare
#pragma unroll 1
                for (int k = 0; k < kB; ++k) {
                    uint32_t ok = 0u;
#pragma unroll
                    for (int x = 0; x < kB; ++x) ok = x == k ? open[x] : ok;
                    if (dc_open_verdicts<T, D, NW, GP>(p, u, G, k_begin + base0 + k * NT + tid, ok, eps_a, misc)) imp |= 1u << k;
                }
            }
#pragma unroll
            for (int k = 0; k < kB; ++k) {
                const int base = base0 + k * NT, i = base + tid;
                if (base + warp * 32 >= n_keys) break;        // uniform in the warp
                const int word = (base >> 5) + warp, from_end = n_words - 1 - ((k_begin >> 5) + word);
                const bool on = i < n_keys, im = (imp >> k) & 1u;
                bool kp = false;
                uint32_t wd = 0u;
                if (on) {
                    wd = update_register(wv[k], im, p.w, t);
                    if (CORM_IN_RANGE(k_begin + i < p.C, p.status)) wordu[k_begin + i] = wd;
                    kp = !evict_on || register_needed(wd, p.w, t) || pv[k] > t - p.r;
                }
                const uint32_t ballot = __ballot_sync(0xffffffffu, kp);
                n_imp += __popc(__ballot_sync(0xffffffffu, im));
                n_keep += __popc(ballot);
                if (lane == 0 && CORM_IN_RANGE(word < kMaxWords, p.status)) keep[word] = ballot;
                if (from_end < 32) {
                    if (lane < cs) push_u32(map_rank(smem_addr(misc->tail + from_end), lane), ballot, map_rank(xbar + kDcCounts * 8, lane));
                    const int s0 = (lane & 7) * 4;            // four registers a lane, four blocks at a time
                    uint4 four;
                    four.x = __shfl_sync(0xffffffffu, wd, s0); four.y = __shfl_sync(0xffffffffu, wd, s0 + 1);
                    four.z = __shfl_sync(0xffffffffu, wd, s0 + 2); four.w = __shfl_sync(0xffffffffu, wd, s0 + 3);
                    const uint32_t at = smem_addr(tail_regs + (31 - from_end) * 32 + s0);
#pragma unroll 1
                    for (int o = lane >> 3; o < cs; o += 4) push_v4(map_rank(at, o), four, map_rank(xbar + kDcCounts * 8, o));
                }
            }
        }
        __syncwarp();
        if (lane < cs)
            push_2u32(map_rank(smem_addr(&misc->verdicts[rank * NW + warp]), lane), (uint32_t)n_keep | (misc->flags[warp] << 24), (uint32_t)n_imp,
                      map_rank(xbar + kDcCounts * 8, lane));
    }
    // outputs (Eq. 1), while the counts travel
    late |= !mbar_wait_cluster(xbar + kDcOutputs * 8, 0);
    for (int x = pair0 + tid; x < pair1; x += NT) {
        float a0 = 0.f, a1 = 0.f;
#pragma unroll
        for (int y = 0; y < kDcMaxCluster; ++y) {
            if (y >= cs) break;
            const float2 v = outputs[y * pair_cap + (x - pair0)];
            a0 += v.x;
            a1 += v.y;
        }
        const double Z = misc->Zt[x / kHalfD];
        const float o0 = (float)((double)a0 / Z), o1 = (float)((double)a1 / Z);
        if constexpr (kBf16) reinterpret_cast<uint32_t*>(p.out)[(size_t)u * np + x] = (uint32_t)float_to_bf16_bits(o0) | ((uint32_t)float_to_bf16_bits(o1) << 16);
        else reinterpret_cast<float2*>(p.out)[(size_t)u * np + x] = make_float2(o0, o1);
    }
    late |= !mbar_wait_cluster(xbar + kDcCounts * 8, 0);
    int new_len = l, imp_total = 0, n_moved = 0;              // n_moved: row moves of the unit
    // Counts, exact heads, moves; the first block waits for the others'. Returns false if a wait expired.
    auto compact = [&]() -> bool {
        if (__syncthreads_or(late)) return false;             // (and the block's keep bits are there)
        int total = 0, before = 0, mine = 0;                  // kept slots of the unit, of the blocks before this one, of this one
        uint32_t marks = 0u;
#pragma unroll
        for (int y = 0; y < kEnt; ++y) {
            const int e = y * 32 + lane;
            if (e >= cs * NW) break;
            const uint2 v = misc->verdicts[e];
            const int n = (int)(v.x & 0xffffffu);
            total += n;
            before += e / NW < rank ? n : 0;
            mine += e / NW == rank ? n : 0;
            imp_total += (int)v.y;
            marks |= v.x >> 24;
        }
        total = __reduce_add_sync(0xffffffffu, total);
        before = __reduce_add_sync(0xffffffffu, before);
        marks = __reduce_or_sync(0xffffffffu, marks);
        uint32_t tail = lane < n_words ? misc->tail[lane] : 0u; // kept slots of the unit's last words, the last one first
        if (marks) {                                          // the same in every block
            const uint32_t meet = xbar + kDcMeet * 8;
            mine = __reduce_add_sync(0xffffffffu, mine);
            const int mine_imp = __reduce_add_sync(0xffffffffu, lane < NW ? (int)misc->verdicts[rank * NW + lane].y : 0);
            if (tid == 0) { misc->cnt.count = mine; misc->cnt.n_imp = mine_imp; }
            uint32_t phase = 0u;
            late |= !dc_meet(meet, cs, phase);
            late |= !dc_exact_heads<T, D, NW, GP>(p, u, G, t, k_begin, k_end, marks, keep, misc, cs, phase);
            phase += 2u * __popc(marks);
            late |= !dc_meet(meet, cs, phase);
            uint4 pc = make_uint4(0u, 0u, 0u, 0u);
            if (lane < cs) pc = ld_peer_v4(map_rank(smem_addr(&misc->cnt), lane));
            total = __reduce_add_sync(0xffffffffu, (int)pc.x);
            before = __reduce_add_sync(0xffffffffu, lane < rank ? (int)pc.x : 0);
            imp_total = (int)pc.y;
            const int wd = n_words - 1 - lane;
            if (wd >= 0) {                                    // from the block that owns the word: the last one with word_begin <= wd
                const int o = (int)((uint32_t)((wd + 1) * cs - 1) / (uint32_t)n_words);
                tail = ld_peer_u32(map_rank(smem_addr(keep + (wd - word_begin(o, cs))), o));
            }
            late |= !dc_meet(meet, cs, phase);                // a block's shared memory stays until its peers have read it
            if (__syncthreads_or(late)) return false;
        }
        // ---- 3. compaction: kept slots at or above the new length move into the holes below it ----
        // Hole number = evicted slots before it, mover number = kept slots behind it, so both follow from the blocks' counts.
        if (evict_on) new_len = total;
        auto row_of = [&](int slot) -> size_t {
            return pt_u ? page_row(__ldcg(pt_u + (slot >> 5)), slot, p.pool_pages, p.status) : (size_t)u * p.C + (size_t)slot;
        };
        int* holes = reinterpret_cast<int*>(smem + kDcRecBytes) + kMaxWords;    // [kDcListCap] each, behind the keep bits
        int* movers = holes + kDcListCap;
        auto hole_words = [&](int i, uint32_t& m, uint32_t& hm) {               // word i of the block: kept slots, holes
            m = keep[i];
            const int s0 = k_begin + i * 32;
            const uint32_t valid = k_end - s0 >= 32 ? 0xffffffffu : (1u << (k_end - s0)) - 1u;
            const uint32_t below = new_len - s0 >= 32 ? 0xffffffffu : (new_len > s0 ? (1u << (new_len - s0)) - 1u : 0u);
            hm = ~m & valid & below;
            m &= ~below;                                      // kept slots at or above the new length
        };
        auto inclusive_scan = [&](int x) -> int {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const int up = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += up; }
            return x;
        };
        if (new_len < l && l - new_len <= kDcListCap) {
            // The usual step: every block fills its own holes; what moves is in the last words of the unit. A word's bits are
            // listed by a warp at once, a bit per lane (one lane walking through a word's bits took 1-2 us of a step).
            const int nw = (n_keys + 31) >> 5, k_lo = max(0, k_begin - before); // number of the block's first hole
            int n_holes = 0;
            for (int i0 = 0; i0 < nw && k_begin + i0 * 32 < new_len; i0 += 32) {
                uint32_t m = 0u, hm = 0u;
                if (i0 + lane < nw) hole_words(i0 + lane, m, hm);
                const int upto = inclusive_scan(__popc(hm));
#pragma unroll
                for (int y = 0; y < 32; y += NW) {
                    const uint32_t bits = __shfl_sync(0xffffffffu, hm, y + warp);
                    const int end = __shfl_sync(0xffffffffu, upto, y + warp);
                    if ((bits >> lane) & 1u) holes[n_holes + end - __popc(bits >> lane)] = k_begin + (i0 + y + warp) * 32 + lane;
                }
                n_holes += __shfl_sync(0xffffffffu, upto, 31);
            }
            {
                const int first_w = new_len >> 5, my_w = n_words - 1 - lane;     // the unit's words that hold movers: [first_w, n_words)
                uint32_t km = my_w >= first_w ? tail : 0u;
                if (my_w == first_w) km &= ~((1u << (new_len & 31)) - 1u);
                const int upto = inclusive_scan(__popc(km));
                n_moved = __shfl_sync(0xffffffffu, upto, 31);
#pragma unroll
                for (int y = 0; y < 32; y += NW) {            // movers are numbered from the last slot down
                    const uint32_t bits = __shfl_sync(0xffffffffu, km, y + warp);
                    const int at = __shfl_sync(0xffffffffu, upto, y + warp) - __popc(bits & ((2u << lane) - 1u)) - k_lo;
                    if (((bits >> lane) & 1u) && at >= 0 && at < n_holes) movers[at] = (n_words - 1 - y - warp) * 32 + lane;
                }
            }
            __syncthreads();
            const int n = min(n_holes, n_moved - k_lo);
            // mover 0 is the unit's last slot, if it stays: the row that was appended
            const int fresh = n > 0 && movers[0] == l_old ? 1 : 0;
            if (fresh && warp == NW - 1 && CORM_IN_RANGE(holes[0] >= 0 && holes[0] < l, p.status)) {
                constexpr int kChunks = S::kRow / 16;
                const size_t at = row_of(holes[0]) * kChunks;
                for (int c = lane; c < 2 * kChunks; c += 32)
                    (c < kChunks ? reinterpret_cast<uint4*>(p.K) + at + c : reinterpret_cast<uint4*>(p.V) + at + c - kChunks)[0] =
                        *reinterpret_cast<const uint4*>(newrow + c * 16);
            }
            block_move_rows<T, D, NT, 4, false>(reinterpret_cast<T*>(p.K), reinterpret_cast<T*>(p.V), row_of, wordu, posu, movers + fresh, holes + fresh, n - fresh, 0, 1, l, p.status);
            for (int i = tid; i < n; i += NT) {               // registers and positions, a mover per thread
                const int from = movers[i], to = holes[i];
                if (!CORM_IN_RANGE(from >= 0 && from < l && to >= 0 && to < l, p.status)) continue;
                const int32_t pos = from == l_old ? t : __ldcg(posu + from);
                wordu[to] = marks ? __ldcg(wordu + from) : tail_regs[from - tail_slot];        // (exact heads change registers)
                posu[to] = pos;
            }
        } else if (new_len < l) {
            // many: the lists go to scratch and the moves are shared out evenly
            int* gholes = reinterpret_cast<int*>(p.stash + (size_t)u * G * p.C) + (size_t)G * p.C;   // behind the unit's logits
            int* gmovers = gholes + p.C / 2;
            int* prefix = holes;                              // [kMaxWords + 1]
            const int nw = (n_keys + 31) >> 5;
            block_popc_scan<NT>(keep, prefix, nw, misc->scan);
            for (int i = tid; i < nw; i += NT) {
                uint32_t km, hm;
                hole_words(i, km, hm);
                const uint32_t m = keep[i];
                const int s0 = k_begin + i * 32, kb = before + prefix[i];        // kept slots before this word
                if (new_len >= s0 && new_len < s0 + 32 && new_len < k_end)       // how many: evicted slots below the new length
                    p.unit_rec[u] = make_int2(new_len - kb - __popc(m & ~km), 0);
                for (; hm; hm &= hm - 1u) {
                    const int bit = __ffs(hm) - 1, x = s0 + bit - kb - __popc(m & ((1u << bit) - 1u));
                    if (CORM_IN_RANGE(x >= 0 && x < p.C / 2, p.status)) gholes[x] = s0 + bit;
                }
                for (; km; km &= km - 1u) {
                    const int bit = __ffs(km) - 1, x = total - 1 - kb - __popc(m & ((1u << bit) - 1u));
                    if (CORM_IN_RANGE(x >= 0 && x < p.C / 2, p.status)) gmovers[x] = s0 + bit;
                }
            }
            uint32_t phase = marks ? 3u + 2u * __popc(marks) : 0u;
            late = !dc_meet(xbar + kDcMeet * 8, cs, phase);
            if (__syncthreads_or(late)) return false;
            if (tid == 0) misc->n_moved = __ldcg(&p.unit_rec[u].x);
            __syncthreads();
            n_moved = misc->n_moved;
            block_move_rows<T, D, NT>(reinterpret_cast<T*>(p.K), reinterpret_cast<T*>(p.V), row_of, wordu, posu, gmovers, gholes, n_moved, rank, cs, l, p.status);
        }
        // every block's row moves come before released pages and the stamp
        if (pt_u || p.unit_stamp) {
            __syncthreads();
            if (tid == 0) mbar_arrive_peer(map_rank(xbar + kDcDone * 8, 0));
            if (rank == 0) {
                late = !mbar_wait_cluster(xbar + kDcDone * 8, 0);
                if (__syncthreads_or(late)) return false;
            }
        }
        return true;
    };
    if (!compact()) {                                         // (no stamp: the unit's next step must not start on rows that may still move)
        late = true;
        leave(false);
        return;
    }
    if (rank != 0) return;
    if (pt_u) settle_pages<NT>(p.page_table, p.page_bits, p.page_room, p.pool_pages, p.pt_stride, p.U, u, l_old, new_len);
    if (pt_u && p.unit_stamp) __syncthreads();
    if (warp == 0) imp_total = __reduce_add_sync(0xffffffffu, imp_total);
    if (tid == 0) {
        p.live_out[u] = new_len;
        publish_unit_stamp(p, u, new_len);
        report_live(p, u, p.step + 1, new_len);
        atomicAdd(p.counters + CNT_APPENDED, 1ull);
        atomicAdd(p.counters + CNT_ATTENDED, (unsigned long long)l);
        if (imp_total) atomicAdd(p.counters + CNT_IMPORTANT, (unsigned long long)imp_total);
        if (new_len < l) atomicAdd(p.counters + CNT_EVICTED, (unsigned long long)(l - new_len));
        if (n_moved) atomicAdd(p.counters + CNT_MOVED, (unsigned long long)n_moved);
    }
}

// One layer's (or, from it on, all layers') K or V storage as a 2-D tensor [rows][D] with boxes of 16 rows x 128 bytes and
// the 128-byte swizzle. The map only ever covers memory of the cache's own device.
inline corm_status_t make_row_tensor_map(CUtensorMap* out, void* base, unsigned long long rows, int D, bool bf16) {
    typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                 const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const EncodeFn encode = [] {                       // looked up once per process
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
            (void)cudaGetLastError();
            fn = nullptr;
        }
        return reinterpret_cast<EncodeFn>(fn);
    }();
    if (!encode) return CORM_ERR_UNSUPPORTED;
    const int e = bf16 ? 2 : 4;
    const cuuint64_t dims[2] = {(cuuint64_t)D, rows};
    const cuuint64_t strides[1] = {(cuuint64_t)(D * e)};
    const cuuint32_t box[2] = {(cuuint32_t)(128 / e), kDcKeys};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = encode(
        out, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, estr,
        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? CORM_OK : CORM_ERR_CUDA;
}

// Warps per block: eight where rows are short (units of a few hundred keys get more warps from eight blocks), four for
// fp32, whose tiles are twice as large (20 units x 250 keys 23 -> 15 us per step).
template <typename T> constexpr int dc_warps() { return Elem<T>::kBytes == 4 ? 4 : 8; }

template <typename T, int D, int GP>
inline corm_status_t launch_decode_cluster_as(DecodeClusterParams& dp, const CUtensorMap& kmap, const CUtensorMap& vmap, int upper,
                                              int tune_split_len, int sm_count, cudaStream_t st) {
    constexpr int NW = dc_warps<T>();
    const DecodeParams& p = dp.p;
    const int sms = sm_count > 0 ? sm_count : 148;
    constexpr int kBlocks = dc_blocks<T, D, GP, NW>();
    // as many blocks per unit as fill the resident slots once, but at least two 32-slot words each ...
    long long cs = (long long)sms * kBlocks / p.U;
    if (tune_split_len) cs = (upper + tune_split_len - 1) / tune_split_len;
    if (cs > (upper + 63) / 64) cs = (upper + 63) / 64;
    // ... and no more words than a block can keep track of
    constexpr int kMaxWords = dc_max_words<T, D, GP, NW>();
    const long long least = ((p.C + 31) / 32 + kMaxWords - 1) / kMaxWords;
    cs = std::max(std::max(cs, least), 1ll);
    if (cs > kDcMaxCluster) cs = kDcMaxCluster;
    if (least > kDcMaxCluster) return CORM_ERR_UNSUPPORTED;
    const int base = dc_smem_layout<T, D, GP, NW>(0).total;
    // Room for logits: what is left of 164 KB per SM where that holds the rest, so that 92 KB of L1 stay for the logits that
    // go through memory and for spilled registers (with 228 KB per SM taken: 128 units x 2800 keys, G 4, 58.7 us a step
    // against 55.4, 32 units x 21400 keys 90.0 against 82.4), otherwise of everything.
    const int budget = (base + 4096 <= 164 * 1024 / kBlocks - 1024 ? 164 : 228) * 1024 / kBlocks - 1024;
    const int need = (int)std::min<long long>(((upper + 31) / 32 + cs - 1) / cs * 32 * (long long)dp.G, 1 << 20);
    dp.lcap = std::max(0, std::min(need, (budget - base) / 128 * 32));
    const size_t smem = (size_t)dc_smem_layout<T, D, GP, NW>(dp.lcap).total;
    auto kern = decode_cluster_kernel<T, D, GP, NW>;
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), (size_t)std::max(budget, base));
    if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)p.U, (unsigned)cs);
        cfg.blockDim = dim3(NW * 32);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1;
        attr[0].val.clusterDim.y = (unsigned)cs;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // set-up overlaps the previous launch's tail
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        e = cudaLaunchKernelEx(&cfg, kern, dp, kmap, vmap);
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    if (e != cudaSuccess) { std::fprintf(stderr, "corm: decode launch: %s\n", cudaGetErrorString(e)); return CORM_ERR_CUDA; }
    return CORM_OK;
}

inline corm_status_t launch_decode_cluster(DecodeClusterParams& dp, bool bf16, int D, const CUtensorMap& kmap, const CUtensorMap& vmap,
                                           int upper, int tune_split_len, int sm_count, cudaStream_t st) {
    const int G = dp.G;
#define CORM_DC(TT, DD, GG) return launch_decode_cluster_as<TT, DD, GG>(dp, kmap, vmap, upper, tune_split_len, sm_count, st)
    if (bf16) {
        if (D == 128) { if (G <= 2) CORM_DC(bf16_t, 128, 2); if (G == 4) CORM_DC(bf16_t, 128, 4); if (G == 8) CORM_DC(bf16_t, 128, 8); }
        else { if (G <= 2) CORM_DC(bf16_t, 64, 2); if (G == 4) CORM_DC(bf16_t, 64, 4); if (G == 8) CORM_DC(bf16_t, 64, 8); }
    } else {
        if (D == 128) { if (G == 1) CORM_DC(float, 128, 1); if (G == 2) CORM_DC(float, 128, 2); if (G == 4) CORM_DC(float, 128, 4); if (G == 8) CORM_DC(float, 128, 8); }
        else { if (G == 1) CORM_DC(float, 64, 1); if (G == 2) CORM_DC(float, 64, 2); if (G == 4) CORM_DC(float, 64, 4); if (G == 8) CORM_DC(float, 64, 8); }
    }
#undef CORM_DC
    return CORM_ERR_UNSUPPORTED;
}

}  // namespace corm
