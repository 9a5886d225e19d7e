// Prompt-end pass: one launch, a thread-block cluster per unit (sequence x kv head), any dtype, head_dim and group.
//
// The min(P, w) recorded queries of the unit's G heads are R = w G "rows"; every row needs the log-sum-exp of its causal
// attention row (Eq. 2) before any verdict (Definition 3.1) can be taken. The cluster's blocks share the unit's keys
// (whole 32-key words each) and go through
//   A. logits of every row against the block's keys, summed as exp(s) per row (fp64, no running maximum: |s| below 650
//      cannot overflow; anything larger sends the unit through the exact path below);
//   -- the blocks exchange their sums through distributed shared memory: one threshold per row
//   B. verdicts of the block's keys for every row -> verdict registers;
//   -- the blocks exchange their counts of surviving keys
//   C. every block gathers its own survivors (K, V rows, registers, positions) to their place in token order.
// Keys stream through a ring of shared-memory buffers of 128 keys (asynchronous copies, two buffers ahead); a block
// whose keys fit the ring reads K once, otherwise phase B finds it in L2 (a unit's K is a few MB and only as many units
// are in flight as fit the machine).
//
// bf16: both contractions run on the tensor cores. Phase A needs fp64-grade logits: operands cut into exact pieces
// (corm_mma.cuh), 7 mma.m16n8k16 per 16 channels for 16 keys x 8 rows. Phase B only has to place a logit on one side of
// its threshold: one plain mma per 16 channels, whose rounding is at most 2^-23 per term; the few logits inside that
// bound are formed again in fp64 by the whole warp (counted in corm_stats_t.near_threshold). If such a logit falls
// within the error of phase A's log-sum-exp itself, it is left undecided and the row is marked; after phase B the
// cluster forms the marked rows' log-sum-exps and verdicts again entirely in fp64 (about one row in 10^4..10^5). So
// every verdict is the fp64 one.
// fp32: fp64 arithmetic on the CUDA cores, lane = key, 4 rows at a time; only ties (1e-13) go to the exact rows, whose
// sums keep the largest logit apart, so that a query at position 1 stays exactly on its threshold.
//
// What bounds it: for windows of a few queries HBM and the latency of the gather (K once, the survivors' V in, K and V
// out); for wide windows the tensor pipe's mma.sync rate in phase A (R P d multiply-adds, seven times).
// Measured against the two-launch pass this replaces (fp64 logits on the CUDA cores; one block per unit gathering) and,
// for fp32 or 64 channels, a pass with one block per unit; us, w = queries in the window, G = heads per group:
//   1024 units x 3250 keys, G 1, w 8    1597 -> 1033      128 units x 3390 keys, G 1, w 256    5341 -> 1735
//   128 units x 8192 keys, G 4, w 8     1821 ->  785      32 units x 8192 keys, G 4, w 128     6736 -> 2235
//   32 units x 32768 keys, G 4, w 16    4618 -> 2363      32 units x 4096 keys, G 1, w 8        259 ->   77
//   fp32: 20 units x 1300 keys, G 2     2787 ->  111      64 channels: 128 units x 2000, G 4  11037 ->  287
#pragma once

#include "corm_fast.cuh"
#include "corm_mma.cuh"

namespace corm {

constexpr int kPcThreads = 256;
constexpr int kPcWarps = kPcThreads / 32;
constexpr int kPcKeys = 128;                    // keys per ring buffer
template <typename T, int D> __host__ __device__ constexpr int pc_bufs() { return D * Elem<T>::kBytes <= 256 ? 3 : 2; }
constexpr int kPcMaxCluster = 8;
constexpr double kPcLogitLimit = 650.0;         // exp of anything below stays finite in fp64, also summed over 2^19 keys

struct PromptClusterParams {
    PromptParams p;
    int32_t log2g;
    int32_t rows8;           // w G rounded up to a multiple of 8
};

struct PcSmem { int ring, zs, thr, n1, qe, flags, words, list, stage, misc, total; };
struct PcMisc {
    double red[kPcWarps][2];
    double mz[2];
    int count, bad, warp_sum[kPcWarps], fail;
    uint32_t amax;                              // largest magnitude (bf16 bits) of the block's keys
    uint16_t tile_amax[3 * kPcKeys / 16];       // ... of every 16-key tile in the ring
};
template <typename T, int D>
__host__ __device__ inline PcSmem pc_smem_layout(int rows8) {
    PcSmem s{};
    int off = 0;
    auto take = [&](int bytes) { int at = off; off = (off + bytes + 127) / 128 * 128; return at; };
    s.ring = take(pc_bufs<T, D>() * kPcKeys * D * Elem<T>::kBytes);
    s.zs = take((rows8 > 64 ? rows8 : 64) * 8);
    s.thr = take(rows8 * 8);
    s.n1 = take(rows8 * 4);
    s.qe = take(rows8 * 4);
    s.flags = take((rows8 + 31) / 32 * 4);
    s.words = take(kPcKeys * 4);
    s.list = take(kPcWarps * 32);               // gather: the kept lanes of a warp's word
    s.stage = take(Elem<T>::kBytes == 4 ? kPcWarps * 4 * D * 8 : 0);
    s.misc = take((int)sizeof(PcMisc));
    s.total = off;
    return s;
}

// byte offset of 16-byte chunk c of row r inside a ring buffer (rows of D elements, chunk index XOR row mod 8)
template <typename T, int D> __device__ __forceinline__ int pc_offset(int r, int c) { return r * (D * Elem<T>::kBytes) + ((c ^ (r & 7)) << 4); }

__device__ __forceinline__ void cp_async16_zfill(uint32_t dst_smem, const void* src_gmem, bool on) {
    const int n = on ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst_smem), "l"(src_gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One logit before the 1/sqrt(d), in fp64, by a whole warp.
template <typename T, int D>
__device__ __forceinline__ double warp_exact_dot(const T* q, const T* k, int lane) {
    constexpr int NPL = D / 32;
    float a[NPL], b[NPL];
    load_slice<T, NPL>(q + lane * NPL, a);
    load_slice<T, NPL>(k + lane * NPL, b);
    double part = 0.0;
#pragma unroll
    for (int i = 0; i < NPL; ++i) part = fma((double)a[i], (double)b[i], part);
    return warp_sum(part);
}

// What the rows of a unit look like: row r = (rho << log2g) + g is the query of window slot rho, head g, at position
// P - (w - 1 - rho); it exists iff rho >= w - min(P, w).
struct PcRows {
    int rows, log2g, w, P;
    __device__ __forceinline__ int rho(int r) const { return r >> log2g; }
    __device__ __forceinline__ int pos(int r) const {       // 0: no such query
        const int x = rho(r), i = P - (w - 1 - x);
        return r < rows && i >= 1 ? i : 0;
    }
    template <typename T, int D> __device__ __forceinline__ const T* q(const T* q_unit, int r) const {
        return q_unit + ((size_t)(r & ((1 << log2g) - 1)) * w + rho(r)) * D;
    }
};

// A verdict's entry in a key's register: the shift register's bit, or the query's position for wide windows.
__device__ __forceinline__ uint32_t pc_mark(int w, int rho, int qpos) { return w <= 32 ? 1u << (w - 1 - rho) : (uint32_t)qpos; }
__device__ __forceinline__ uint32_t pc_join(int w, uint32_t a, uint32_t b) { return w <= 32 ? (a | b) : max(a, b); }

// The marked rows, exactly: log-sum-exp with a running maximum and every verdict in fp64 straight from global memory.
// Rare (or asked for by an inflated bound); all blocks of the cluster take it together. Verdicts that phase B was sure
// of hold for the exact threshold too, so adding marks is enough.
template <typename T, int D>
__device__ __noinline__ void pc_exact_rows(const PromptParams& p, const PcRows& R, const T* Qu, const T* Ku, int k_begin, int k_end,
                                           const uint32_t* flags, uint32_t* words_g, PcMisc* misc, int cs) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double inv_root_d = inv_root_dim(D);
    const uint32_t mz_addr = smem_addr(misc->mz);
    for (int r = 0; r < R.rows; ++r) {
        if (!((flags[r >> 5] >> (r & 31)) & 1u)) continue;
        const int qpos = R.pos(r);
        if (!qpos) continue;
        const T* qr = R.q<T, D>(Qu, r);
        const int end = min(k_end, qpos);                     // causal row: keys 1..position of the query
        double m = -INFINITY, Z = 0.0;
        for (int j = k_begin + warp; j < end; j += kPcWarps) {
            const double s = warp_exact_dot<T, D>(qr, Ku + (size_t)j * D, lane) * inv_root_d;
            if (s > m) { Z = Z * exp(m - s) + 1.0; m = s; }
            else Z += exp(s - m);
        }
        if (lane == 0) { misc->red[warp][0] = m; misc->red[warp][1] = Z; }
        __syncthreads();
        if (tid == 0) {
            double mb = -INFINITY, Zb = 0.0;
            for (int x = 0; x < kPcWarps; ++x) mb = fmax(mb, misc->red[x][0]);
            for (int x = 0; x < kPcWarps; ++x)
                if (misc->red[x][1] > 0.0) Zb += misc->red[x][1] * exp(misc->red[x][0] - mb);
            misc->mz[0] = mb; misc->mz[1] = Zb;
        }
        cluster_sync();
        double M = -INFINITY, Zt = 0.0;
        for (int x = 0; x < cs; ++x) M = fmax(M, ld_peer_f64(map_rank(mz_addr, x)));
        for (int x = 0; x < cs; ++x) {
            const double z = ld_peer_f64(map_rank(mz_addr + 8, x));
            if (z > 0.0) Zt += z * exp(ld_peer_f64(map_rank(mz_addr, x)) - M);
        }
        const double thr = M + log(Zt) + p.log_alpha - log((double)qpos);
        for (int j = k_begin + warp; j < end; j += kPcWarps) {
            const double s = warp_exact_dot<T, D>(qr, Ku + (size_t)j * D, lane) * inv_root_d;
            if (lane == 0 && s >= thr) words_g[j] = pc_join(p.w, words_g[j], pc_mark(p.w, R.rho(r), qpos));
        }
        cluster_sync();                                       // everybody has read mz
    }
}

// Query pieces of 8 rows in the B operand's layout (row n = lane / 4), held in registers.
template <int D> struct PcFrag { uint32_t b1[D / 16][2], b2[D / 16][2], b3[D / 16][2]; };

template <int D>
__device__ __forceinline__ void pc_load_raw(const PcRows& R, const bf16_t* Qu, int octet, int lane, uint32_t (&raw)[D / 16][2]) {
    const int r = 8 * octet + (lane >> 2);
    const bool on = R.pos(r) > 0;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(R.q<bf16_t, D>(Qu, on ? r : R.rows - 1)) + (lane & 3);
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
        raw[kk][0] = on ? __ldg(src + kk * 8) : 0u;
        raw[kk][1] = on ? __ldg(src + kk * 8 + 4) : 0u;
    }
}

// The pieces, and the row's norms for the error bounds. Returns false if the row leaves the safe range.
template <int D>
__device__ __forceinline__ bool pc_load_frag(const PcRows& R, const bf16_t* Qu, int octet, int lane, PcFrag<D>& f, float* n1_sm, float* qe_sm) {
    uint32_t raw[D / 16][2];
    pc_load_raw<D>(R, Qu, octet, lane, raw);
    uint32_t mx = 0u;
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) { mx = max_abs_bf16x2(mx, raw[kk][0]); mx = max_abs_bf16x2(mx, raw[kk][1]); }
    uint32_t m16 = max(mx & 0xffffu, mx >> 16);
    m16 = max(m16, __shfl_xor_sync(0xffffffffu, m16, 1));
    m16 = max(m16, __shfl_xor_sync(0xffffffffu, m16, 2));
    const bool ok = m16 < kSplitMaxBits;
    const float c = split_query_const(ok ? __uint_as_float(m16 << 16) : 1.f);
    float n1 = 0.f, n2 = 0.f, n3 = 0.f;
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float a[2] = {__uint_as_float(raw[kk][h] << 16), __uint_as_float(raw[kk][h] & 0xffff0000u)}, x1[2], x2[2], x3[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                split_query(a[e], c, x1[e], x2[e], x3[e]);
                n1 += fabsf(a[e]); n2 += fabsf(x2[e]); n3 += fabsf(x3[e]);
            }
            f.b1[kk][h] = (__float_as_uint(x1[0]) >> 16) | (__float_as_uint(x1[1]) & 0xffff0000u);   // exact: bf16 numbers
            f.b2[kk][h] = (__float_as_uint(x2[0]) >> 16) | (__float_as_uint(x2[1]) & 0xffff0000u);
            f.b3[kk][h] = (__float_as_uint(x3[0]) >> 16) | (__float_as_uint(x3[1]) & 0xffff0000u);
        }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        n1 += __shfl_xor_sync(0xffffffffu, n1, o);
        n2 += __shfl_xor_sync(0xffffffffu, n2, o);
        n3 += __shfl_xor_sync(0xffffffffu, n3, o);
    }
    if ((lane & 3) == 0) {                                    // the same values from every warp that holds the octet
        n1_sm[8 * octet + (lane >> 2)] = n1 * 1.0001f;
        qe_sm[8 * octet + (lane >> 2)] = split_error(n1, n2, n3);
    }
    return ok;
}

template <typename T, int D>
__global__ void __launch_bounds__(kPcThreads, (D * Elem<T>::kBytes <= 256) ? 2 : 1)
prompt_cluster_kernel(const __grid_constant__ PromptClusterParams pp) {
    extern __shared__ __align__(128) unsigned char smem[];
    const PromptParams& p = pp.p;
    constexpr bool kBf16 = Elem<T>::kBytes == 2;
    constexpr int kRow = D * Elem<T>::kBytes, kChunks = kRow / 16;
    constexpr int kRowUnit = kBf16 ? 8 : 4;                   // rows a warp works on at a time
    constexpr int kKeyUnit = kBf16 ? 16 : 32;                 // keys
    constexpr int kSubs = kPcKeys / kKeyUnit;                 // key units per buffer
    constexpr int kBufs = pc_bufs<T, D>();
    const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cs = (int)cluster_size(), rank = (int)cluster_rank();
    asm volatile("griddepcontrol.wait;" ::: "memory");        // prompt_begin_kernel, and what precedes it on the stream
    const int b = u / p.Hkv, P = __ldcg(p.prompt_lens + b), w = p.w, wp = min(P, w);
    if (P > p.C) {
        if (rank == 0 && tid == 0) { report_status(p.status, CORM_ERR_CAPACITY); p.live_out[u] = 0; }
        return;
    }
    if (P == 0) {
        if (rank == 0 && tid == 0) {
            p.live_out[u] = 0; report_live(p, u, 0, 0);
            if (p.page_table) {  // an empty unit still owns the page its first append goes to
                const int pg = claim_page(p.page_bits, p.pool_pages, p.U, u, 0);
                p.page_table[(size_t)u * p.pt_stride] = pg + 1;
                p.page_room[u] = pg >= 0;
            }
        }
        return;
    }
    const PcSmem lay = pc_smem_layout<T, D>(pp.rows8);
    double* zs = reinterpret_cast<double*>(smem + lay.zs);
    double* thr_sm = reinterpret_cast<double*>(smem + lay.thr);
    float* n1_sm = reinterpret_cast<float*>(smem + lay.n1);
    float* qe_sm = reinterpret_cast<float*>(smem + lay.qe);
    uint32_t* flags = reinterpret_cast<uint32_t*>(smem + lay.flags);
    uint32_t* words_sm = reinterpret_cast<uint32_t*>(smem + lay.words);
    PcMisc* misc = reinterpret_cast<PcMisc*>(smem + lay.misc);

    const PcRows R{w << pp.log2g, pp.log2g, w, P};
    const int n_words = (P + 31) >> 5;
    const int w0 = (int)((long long)n_words * rank / cs), w1 = (int)((long long)n_words * (rank + 1) / cs);
    uint32_t* keep_g = p.keepmask + (size_t)u * keepmask_words(p.C) + w0;            // the block's keep bits
    const int k_begin = w0 * 32, k_end = min(P, w1 * 32), n_keys = max(0, k_end - k_begin);
    const int nc = (n_keys + kPcKeys - 1) / kPcKeys;
    const bool resident = nc <= kBufs;
    const T* Ku = reinterpret_cast<const T*>(p.k_prompt) + (size_t)u * p.p_max * D;
    const T* Vu = reinterpret_cast<const T*>(p.v_prompt) + (size_t)u * p.p_max * D;
    const T* Qu = reinterpret_cast<const T*>(p.q_last) + ((size_t)u << pp.log2g) * w * D;
    uint32_t* words_g = reinterpret_cast<uint32_t*>(p.stash) + (size_t)u * p.C;      // scratch registers of this unit
    const double inv_root_d = inv_root_dim(D), root_d = D == 128 ? 11.313708498984760390 : 8.0;
    const uint32_t ring = smem_addr(smem + lay.ring);

    auto issue = [&](int c) {                                 // chunk c of the block's keys -> its ring buffer
        if (c < nc) {
            const uint32_t dst = ring + (c % kBufs) * (kPcKeys * kRow);
            const unsigned char* src = reinterpret_cast<const unsigned char*>(Ku + (size_t)(k_begin + c * kPcKeys) * D);
            const int valid = n_keys - c * kPcKeys;
#pragma unroll 4
            for (int x = tid; x < kPcKeys * kChunks; x += kPcThreads) {
                const int r = x / kChunks, ch = x % kChunks;
                const bool on = r < valid;
                cp_async16_zfill(dst + pc_offset<T, D>(r, ch), src + (on ? (size_t)r * kRow + ch * 16 : 0), on);
            }
        }
        cp_async_commit();
    };
    auto measure = [&](int c) {                               // largest magnitude of every 16-key tile of a buffer (warp = tile)
        const unsigned char* buf = smem + lay.ring + (c % kBufs) * (kPcKeys * kRow);
        uint32_t m = 0u;
#pragma unroll
        for (int x = 0; x < kChunks / 2; ++x) {
            const uint4 v = *reinterpret_cast<const uint4*>(buf + warp * 16 * kRow + (x * 32 + lane) * 16);
            m = max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(m, v.x), v.y), v.z), v.w);
        }
        m = __reduce_max_sync(0xffffffffu, max(m & 0xffffu, m >> 16));
        if (lane == 0) { misc->tile_amax[(c % kBufs) * (kPcKeys / 16) + warp] = (uint16_t)m; atomicMax(&misc->amax, m); }
    };
#pragma unroll
    for (int i = 0; i < kBufs - 1; ++i) issue(i);
    for (int i = tid; i < (pp.rows8 + 31) / 32; i += kPcThreads) flags[i] = 0u;
    if (tid == 0) { misc->bad = 0; misc->amax = 0u; misc->fail = 0; }

    // who works on what: warps own row units where there are at least as many, otherwise they share them by key units
    const int n_ru = (R.rows + kRowUnit - 1) / kRowUnit;
    int ru_slots = 1;                                         // warps side by side over the row units (a power of two)
    while (ru_slots < n_ru && ru_slots < kPcWarps) ru_slots *= 2;
    const int key_groups = min(kPcWarps / ru_slots, kSubs);
    const int my_ru = warp % ru_slots, my_kg = warp / ru_slots;
    const bool works = my_ru < n_ru && my_kg < key_groups;
    const bool keep_rows = n_ru <= ru_slots;                  // a warp has one row unit at most: its pieces stay in registers

    // ---- A. sums of exp(s) per row ----
    bool bad = false;
    {
        PcFrag<kBf16 ? D : 16> f;
        double z[4] = {0.0, 0.0, 0.0, 0.0};                   // bf16: rows 2 (lane % 4), + 1 of the octet; fp32: the four rows
        double* qst = reinterpret_cast<double*>(smem + lay.stage) + warp * 4 * D;      // fp32: the rows as doubles
        for (int i = tid; i < max(pp.rows8, 64); i += kPcThreads) zs[i] = 0.0;
        auto fold = [&](int ru) {                             // the warp's lanes -> its slots of zs
            if constexpr (kBf16) {
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) { z[0] += __shfl_xor_sync(0xffffffffu, z[0], o); z[1] += __shfl_xor_sync(0xffffffffu, z[1], o); }
                if (lane < 4) {
                    double* dst = zs + my_kg * (n_ru * kRowUnit) + ru * kRowUnit + 2 * lane;
                    dst[0] += z[0]; dst[1] += z[1];
                }
            } else {
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const double t = warp_sum(z[x]);
                    if (lane == 0) zs[my_kg * (n_ru * kRowUnit) + ru * kRowUnit + x] += t;
                }
            }
            z[0] = z[1] = z[2] = z[3] = 0.0;
        };
        bool have = false;
        for (int c = 0; c < nc; ++c) {
            cp_async_wait<kBufs - 2>();
            __syncthreads();                                  // chunk c is in; everybody is done with chunk c - 1
            issue(c + kBufs - 1);
            const unsigned char* buf = smem + lay.ring + (c % kBufs) * (kPcKeys * kRow);
            if constexpr (kBf16) { measure(c); __syncthreads(); }
            const int n_valid = min(kPcKeys, n_keys - c * kPcKeys);
            if (works)
                for (int ru = my_ru; ru < n_ru; ru += ru_slots) {
                    if (!keep_rows || !have) {
                        if constexpr (kBf16) {
                            bad |= !pc_load_frag<D>(R, Qu, ru, lane, f, n1_sm, qe_sm);
                        } else {
                            __syncwarp();
                            for (int x = lane; x < 4 * D; x += 32) {
                                const int r = ru * 4 + x / D;
                                qst[x] = R.pos(r) ? (double)Elem<T>::load(R.q<T, D>(Qu, r) + x % D) : 0.0;
                            }
                            __syncwarp();
                        }
                        have = true;
                    }
                    const int r0 = ru * kRowUnit + (kBf16 ? 2 * (lane & 3) : 0);
                    int qpos[kBf16 ? 2 : 4];
#pragma unroll
                    for (int x = 0; x < (kBf16 ? 2 : 4); ++x) qpos[x] = R.pos(r0 + x);
                    for (int sub = my_kg; sub < kSubs && sub * kKeyUnit < n_valid; sub += key_groups) {
                        const int j0 = k_begin + c * kPcKeys + sub * kKeyUnit;       // 0-based key index
                        if constexpr (kBf16) {
                            const SplitGrid g = split_grid(misc->tile_amax[(c % kBufs) * (kPcKeys / 16) + sub]);
                            float hi[4] = {0.f, 0.f, 0.f, 0.f}, mid[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
                            const uint32_t arow = ring + (c % kBufs) * (kPcKeys * kRow) + (sub * 16 + (lane & 15)) * kRow;
#pragma unroll
                            for (int kk = 0; kk < D / 16; ++kk) {
                                uint32_t a[4], k1[4], k2[4], r2[4];
                                ldmatrix_x4(a, arow + (((kk * 2 + (lane >> 4)) ^ (lane & 7)) << 4));
                                split_key(a, g, k1, k2, r2);
                                float t[4] = {0.f, 0.f, 0.f, 0.f};
                                mma16816(hi, k1, f.b1[kk][0], f.b1[kk][1]);
                                mma16816(mid, k1, f.b2[kk][0], f.b2[kk][1]);
                                mma16816(t, k2, f.b2[kk][0], f.b2[kk][1]);
                                mma16816(mid, k2, f.b1[kk][0], f.b1[kk][1]);
                                mma16816(t, r2, f.b1[kk][0], f.b1[kk][1]);
                                mma16816(t, r2, f.b2[kk][0], f.b2[kk][1]);
                                mma16816(t, k1, f.b3[kk][0], f.b3[kk][1]);
#pragma unroll
                                for (int x = 0; x < 4; ++x) lo[x] += t[x];
                            }
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                const int j = j0 + (lane >> 2) + (x >> 1) * 8;
                                const double s = (((double)hi[x] + (double)mid[x]) + (double)lo[x]) * inv_root_d;
                                const bool on = j < k_end && j < qpos[x & 1];           // causal row: keys 1..position of the query
                                bad |= on && !(fabs(s) < kPcLogitLimit);
                                z[x & 1] += on ? exp_nonpos(s) : 0.0;
                            }
                        } else {
                            double acc[4] = {0.0, 0.0, 0.0, 0.0};
                            const int kr = sub * 32 + lane;
#pragma unroll 4
                            for (int ch = 0; ch < kChunks; ++ch) {
                                const float4 kv = *reinterpret_cast<const float4*>(buf + pc_offset<T, D>(kr, ch));
                                const double k4[4] = {(double)kv.x, (double)kv.y, (double)kv.z, (double)kv.w};
#pragma unroll
                                for (int x = 0; x < 4; ++x) {
                                    const double2 qa = *reinterpret_cast<const double2*>(qst + x * D + ch * 4);
                                    const double2 qb = *reinterpret_cast<const double2*>(qst + x * D + ch * 4 + 2);
                                    acc[x] = fma(qa.x, k4[0], acc[x]); acc[x] = fma(qa.y, k4[1], acc[x]);
                                    acc[x] = fma(qb.x, k4[2], acc[x]); acc[x] = fma(qb.y, k4[3], acc[x]);
                                }
                            }
                            const int j = j0 + lane;
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                const double s = acc[x] * inv_root_d;
                                const bool on = j < k_end && j < qpos[x];
                                bad |= on && !(fabs(s) < kPcLogitLimit);
                                z[x] += on ? exp_nonpos(s) : 0.0;
                            }
                        }
                    }
                    if (!keep_rows) fold(ru);
                }
        }
        __syncthreads();
        if (works && keep_rows) fold(my_ru);
        if constexpr (kBf16)                                  // a block without keys has no pieces yet, but the norms are asked for
            if (nc == 0 && works) for (int ru = my_ru; ru < n_ru; ru += ru_slots) pc_load_frag<D>(R, Qu, ru, lane, f, n1_sm, qe_sm);
    }
    if (bad) misc->bad = 1;
    __syncthreads();
    if (kBf16 && tid == 0 && misc->amax >= kSplitMaxBits) misc->bad = 1;
    for (int i = tid; i < n_ru * kRowUnit; i += kPcThreads)   // key groups of this block, in a fixed order
        for (int x = 1; x < key_groups; ++x) zs[i] += zs[x * (n_ru * kRowUnit) + i];
    cluster_sync();

    // ---- thresholds of Definition 3.1 in log form: s >= lse + ln(alpha) - ln(position of the query) ----
    int any_bad = 0;
    uint32_t amax_unit = 0u;
    for (int x = 0; x < cs; ++x) {
        any_bad |= (int)ld_peer_u32(map_rank(smem_addr(&misc->bad), x));
        amax_unit = max(amax_unit, ld_peer_u32(map_rank(smem_addr(&misc->amax), x)));
    }
    for (int r = tid; r < n_ru * kRowUnit; r += kPcThreads) {
        const int qpos = R.pos(r);
        double Z = 0.0;
        for (int x = 0; x < cs; ++x) Z += ld_peer_f64(map_rank(smem_addr(zs + r), x));
        thr_sm[r] = qpos ? log(Z) + p.log_alpha - log((double)qpos) : INFINITY;
        if (any_bad && qpos) atomicOr(flags + (r >> 5), 1u << (r & 31));      // every row of the unit goes through the exact path
    }
    // error of a threshold per unit of qe (every logit of the row is off by at most this much, so its log-sum-exp is too)
    const double eps_unit = kBf16 ? p.bound_scale * (double)split_amax(amax_unit) * inv_root_d : 0.0;

    // ---- B. verdicts -> registers ----
    if (!resident) {
#pragma unroll
        for (int i = 0; i < kBufs - 1; ++i) issue(i);
    }
    for (int c = 0; c < nc; ++c) {
        if (!resident) cp_async_wait<kBufs - 2>();
        if (tid < kPcKeys) words_sm[tid] = 0u;
        __syncthreads();
        if (!resident) {
            issue(c + kBufs - 1);
            if constexpr (kBf16) { measure(c); __syncthreads(); }
        }
        const unsigned char* buf = smem + lay.ring + (c % kBufs) * (kPcKeys * kRow);
        const int n_valid = min(kPcKeys, n_keys - c * kPcKeys);
        if (works && !any_bad)
            for (int ru = my_ru; ru < n_ru; ru += ru_slots) {
                if constexpr (kBf16) {
                    uint32_t q[D / 16][2];
                    pc_load_raw<D>(R, Qu, ru, lane, q);
                    const int r0 = ru * 8 + 2 * (lane & 3);
                    float thr_f[2], err_f[2], slack[2];
                    int qpos[2];
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        qpos[x] = R.pos(r0 + x);
                        thr_f[x] = (float)(thr_sm[r0 + x] * root_d);
                        // D roundings of 2^-23 on sums of at most A |q|_1 (a tenth of slack), the threshold's own rounding,
                        // and the threshold's error
                        err_f[x] = (float)p.bound_scale * ((float)D * 1.1f / 8388608.f * n1_sm[r0 + x]);
                        slack[x] = fabsf(thr_f[x]) * 2.4e-7f + (float)(eps_unit * qe_sm[r0 + x] * root_d) * 1.01f;
                    }
                    for (int sub = my_kg; sub < kSubs && sub * 16 < n_valid; sub += key_groups) {
                        const int j0 = k_begin + c * kPcKeys + sub * 16;
                        const float A = split_amax(misc->tile_amax[(c % kBufs) * (kPcKeys / 16) + sub]);
                        float acc[4] = {0.f, 0.f, 0.f, 0.f};
                        const uint32_t arow = ring + (c % kBufs) * (kPcKeys * kRow) + (sub * 16 + (lane & 15)) * kRow;
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk) {
                            uint32_t a[4];
                            ldmatrix_x4(a, arow + (((kk * 2 + (lane >> 4)) ^ (lane & 7)) << 4));
                            mma16816(acc, a, q[kk][0], q[kk][1]);
                        }
                        uint32_t mark[2] = {0u, 0u};          // keys lane / 4 and lane / 4 + 8
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int j = j0 + (lane >> 2) + (x >> 1) * 8, row = r0 + (x & 1);
                            const bool on = j < k_end && j < qpos[x & 1];
                            const float margin = acc[x] - thr_f[x & 1], err = err_f[x & 1] * A + slack[x & 1];
                            bool imp = on && margin >= err;
                            uint32_t unsure = __ballot_sync(0xffffffffu, on && margin < err && margin > -err);
                            if (unsure && lane == 0) atomicAdd(p.counters + CNT_NEAR, (unsigned long long)__popc(unsure));
                            while (unsure) {                  // formed again in fp64, one after the other, by the whole warp
                                const int src = __ffs(unsure) - 1;
                                unsure &= unsure - 1u;
                                const int js = __shfl_sync(0xffffffffu, j, src), rs = __shfl_sync(0xffffffffu, row, src);
                                const double s = warp_exact_dot<T, D>(R.q<T, D>(Qu, rs), Ku + (size_t)js * D, lane) * inv_root_d;
                                const double th = thr_sm[rs], e = eps_unit * (double)qe_sm[rs] + 1e-13 * (1.0 + fabs(th));
                                if (lane == src) imp = s - th > e;                     // closer than that: left to the exact rows
                                if (lane == 0 && fabs(s - th) <= e) atomicOr(flags + (rs >> 5), 1u << (rs & 31));
                            }
                            if (imp) mark[x >> 1] = pc_join(w, mark[x >> 1], pc_mark(w, R.rho(row), qpos[x & 1]));
                        }
#pragma unroll
                        for (int y = 0; y < 2; ++y) {
                            mark[y] = pc_join(w, mark[y], __shfl_xor_sync(0xffffffffu, mark[y], 1));
                            mark[y] = pc_join(w, mark[y], __shfl_xor_sync(0xffffffffu, mark[y], 2));
                            if ((lane & 3) == 0 && mark[y]) {
                                uint32_t* dst = words_sm + sub * 16 + (lane >> 2) + y * 8;
                                if (w <= 32) atomicOr(dst, mark[y]);
                                else atomicMax(dst, mark[y]);
                            }
                        }
                    }
                } else {
                    double* qst = reinterpret_cast<double*>(smem + lay.stage) + warp * 4 * D;
                    if (!keep_rows) {
                        __syncwarp();
                        for (int x = lane; x < 4 * D; x += 32) {
                            const int r = ru * 4 + x / D;
                            qst[x] = R.pos(r) ? (double)Elem<T>::load(R.q<T, D>(Qu, r) + x % D) : 0.0;
                        }
                        __syncwarp();
                    }
                    for (int sub = my_kg; sub < kSubs && sub * 32 < n_valid; sub += key_groups) {
                        double acc[4] = {0.0, 0.0, 0.0, 0.0};
                        const int kr = sub * 32 + lane, j = k_begin + c * kPcKeys + kr;
#pragma unroll 4
                        for (int ch = 0; ch < kChunks; ++ch) {
                            const float4 kv = *reinterpret_cast<const float4*>(buf + pc_offset<T, D>(kr, ch));
                            const double k4[4] = {(double)kv.x, (double)kv.y, (double)kv.z, (double)kv.w};
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                const double2 qa = *reinterpret_cast<const double2*>(qst + x * D + ch * 4);
                                const double2 qb = *reinterpret_cast<const double2*>(qst + x * D + ch * 4 + 2);
                                acc[x] = fma(qa.x, k4[0], acc[x]); acc[x] = fma(qa.y, k4[1], acc[x]);
                                acc[x] = fma(qb.x, k4[2], acc[x]); acc[x] = fma(qb.y, k4[3], acc[x]);
                            }
                        }
                        uint32_t mark = 0u;
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int row = ru * 4 + x, qpos = R.pos(row);
                            if (j >= k_end || j >= qpos) continue;
                            const double margin = acc[x] * inv_root_d - thr_sm[row], e = 1e-13 * (1.0 + fabs(thr_sm[row]));
                            if (margin > e) mark = pc_join(w, mark, pc_mark(w, R.rho(row), qpos));
                            else if (margin >= -e) atomicOr(flags + (row >> 5), 1u << (row & 31));   // a tie (a query at position 1): the exact rows
                        }
                        if (mark) {
                            if (w <= 32) atomicOr(words_sm + kr, mark);
                            else atomicMax(words_sm + kr, mark);
                        }
                    }
                }
            }
        __syncthreads();
        if (tid < n_valid) words_g[k_begin + c * kPcKeys + tid] = words_sm[tid];
    }
    __syncthreads();

    // ---- keep rule of Algorithm 1 for the block's keys; counts and marked rows are exchanged together ----
    const bool evict_on = wp >= w;
    auto keep_pass = [&]() {
        int mine = 0;
        for (int base = 0; base < n_keys; base += kPcThreads) {
            const int j = k_begin + base + tid;
            bool keep = false;
            if (base + tid < n_keys) keep = !evict_on || register_needed(__ldcg(words_g + j), w, P) || (j + 1) > P - p.r;
            const uint32_t ballot = __ballot_sync(0xffffffffu, keep);
            if (lane == 0 && base + warp * 32 < n_keys) { keep_g[(base >> 5) + warp] = ballot; mine += __popc(ballot); }
        }
        if (lane == 0) misc->warp_sum[warp] = mine;
        __syncthreads();
        if (tid == 0) {
            int t = 0;
            for (int x = 0; x < kPcWarps; ++x) t += misc->warp_sum[x];
            misc->count = t;
        }
    };
    keep_pass();
    cluster_sync();
    bool marked = false;
    for (int i = tid; i < (pp.rows8 + 31) / 32; i += kPcThreads)
        for (int x = 0; x < cs; ++x) marked |= ld_peer_u32(map_rank(smem_addr(flags + i), x)) != 0u;
    if (__syncthreads_or(marked)) {
        cluster_sync();                                       // everybody has looked at everybody's marks
        for (int i = tid; i < (pp.rows8 + 31) / 32; i += kPcThreads) {
            uint32_t m = 0u;
            for (int x = 0; x < cs; ++x) m |= ld_peer_u32(map_rank(smem_addr(flags + i), x));
            thr_sm[i] = __longlong_as_double((long long)m);  // thresholds are done with: parked until every block has read
        }
        cluster_sync();
        for (int i = tid; i < (pp.rows8 + 31) / 32; i += kPcThreads) flags[i] = (uint32_t)__double_as_longlong(thr_sm[i]);
        __syncthreads();
        pc_exact_rows<T, D>(p, R, Qu, Ku, k_begin, k_end, flags, words_g, misc, cs);
        __syncthreads();
        keep_pass();
        cluster_sync();
    }
    int kept_total = 0, first = 0;
    for (int x = 0; x < cs; ++x) {
        const int n = (int)ld_peer_u32(map_rank(smem_addr(&misc->count), x));
        if (x < rank) first += n;
        kept_total += n;
    }
    int32_t* pt_u = p.page_table ? p.page_table + (size_t)u * p.pt_stride : nullptr;
    if (pt_u) {   // the block in whose range a page starts claims it (the last block also the page of the next append)
        const int my_end = first + misc->count;
        const int last_page = min(kept_total / kPageKeys + 1, p.pt_stride);
        const int i0 = rank == 0 ? 0 : (first + kPageKeys - 1) / kPageKeys;
        const int i1 = rank == cs - 1 ? last_page : min(last_page, (my_end + kPageKeys - 1) / kPageKeys);
        for (int i = i0 + tid; i < i1; i += kPcThreads) {
            const int pg = claim_page(p.page_bits, p.pool_pages, p.U, u, i);
            pt_u[i] = pg + 1;
            if (pg < 0) misc->fail = 1;
        }
        __threadfence();
        cluster_sync();
        int failed = 0;
        for (int x = 0; x < cs; ++x) failed |= (int)ld_peer_u32(map_rank(smem_addr(&misc->fail), x));
        if (rank == 0 && tid == 0) p.page_room[u] = failed ? 0 : 1;
        if (failed) {                                         // the pool is too small: the unit is left empty
            if (rank == 0 && tid == 0) { report_status(p.status, CORM_ERR_CAPACITY); p.live_out[u] = 0; report_live(p, u, 0, 0); }
            cluster_sync();
            return;
        }
    }

    // ---- C. ordered gather of the survivors: a warp takes a 32-key word at a time, eight 16-byte pieces per lane in flight ----
    {
        unsigned char* Kl = reinterpret_cast<unsigned char*>(p.K);
        unsigned char* Vl = reinterpret_cast<unsigned char*>(p.V);
        uint32_t* wordu = p.word + (size_t)u * p.C;
        int32_t* posu = p.pos + (size_t)u * p.C;
        const int my_words = (n_keys + 31) / 32;
        unsigned char* list = smem + lay.list + warp * 32;
        int base = 0, done = 0;                               // survivors of the block before word `done` (a part per lane)
        for (int i = warp; i < my_words; i += kPcWarps) {
            for (int x = done + lane; x < i; x += 32) base += __popc(__ldcg(keep_g + x));
            done = i;
            const uint32_t m = __ldcg(keep_g + i);
            const int n = __popc(m), dst0 = first + __reduce_add_sync(0xffffffffu, base), j0 = k_begin + i * 32;
            if ((m >> lane) & 1u) {
                const int k = __popc(m & ((1u << lane) - 1u)), dst = dst0 + k;
                list[k] = (unsigned char)lane;
                wordu[dst] = __ldcg(words_g + j0 + lane);
                posu[dst] = j0 + lane + 1;
            }
            __syncwarp();
            constexpr int kPer = 2 * kChunks;                 // 16-byte pieces of a row pair (K and V)
            constexpr int kFly = 8;
            for (int x0 = 0; x0 < n * kPer; x0 += 32 * kFly) {
                uint4 buf[kFly];
                size_t at[kFly];
#pragma unroll
                for (int y = 0; y < kFly; ++y) {
                    const int x = x0 + y * 32 + lane, k = x / kPer, ch = x % kPer;
                    at[y] = (size_t)-1;
                    if (k < n) {
                        const int src = j0 + list[k], dst = dst0 + k;
                        const size_t row = pt_u ? page_row(__ldcg(pt_u + (dst >> 5)), dst, p.pool_pages, p.status) : (size_t)u * p.C + dst;
                        at[y] = row * kRow + (ch % kChunks) * 16;
                        buf[y] = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned char*>(ch < kChunks ? Ku : Vu) + (size_t)src * kRow) + ch % kChunks);
                    }
                }
#pragma unroll
                for (int y = 0; y < kFly; ++y) {
                    const int ch = (x0 + y * 32 + lane) % kPer;
                    if (at[y] != (size_t)-1) *reinterpret_cast<uint4*>((ch < kChunks ? Kl : Vl) + at[y]) = buf[y];
                }
            }
            __syncwarp();                                     // the list is the next word's
        }
    }
    if (rank == 0 && tid == 0) {
        if (kBf16) p.kmax[u] = amax_unit;
        p.live_out[u] = kept_total;
        report_live(p, u, 0, kept_total);
        atomicAdd(p.counters + CNT_APPENDED, (unsigned long long)P);
        if (kept_total < P) atomicAdd(p.counters + CNT_EVICTED, (unsigned long long)(P - kept_total));
    }
    cluster_sync();                                           // a block's shared memory stays until its peers have read it
}

// First launch of the pass: the sequences' token and row counts (they travel in the launch's parameters) and a clean
// slate for the layer's arrival counters, stamps, statistics and (paged) page tables. One launch of a few microseconds
// where nine small copies and memsets stood before; the pass itself is programmatic-dependent on it.
constexpr int kPbLens = 512;                              // sequences per launch
constexpr int kPbThreads = 256;
struct PromptBeginParams {
    int32_t lens[kPbLens];
    int32_t first, n, w;                                  // sequences [first, first + n)
    int32_t* base_tokens;
    int32_t* base_obs;
    struct Span { uint32_t* ptr; unsigned long long words; } clear[9];    // 32-bit words to zero
};
__global__ void __launch_bounds__(kPbThreads) prompt_begin_kernel(const __grid_constant__ PromptBeginParams p) {
    const unsigned long long at = (unsigned long long)blockIdx.x * kPbThreads + threadIdx.x, step = (unsigned long long)gridDim.x * kPbThreads;
    if (at < (unsigned long long)p.n) {
        p.base_tokens[p.first + at] = p.lens[at];
        p.base_obs[p.first + at] = min(p.lens[at], p.w);
    }
#pragma unroll
    for (int i = 0; i < 9; ++i)
        for (unsigned long long x = at; x < p.clear[i].words; x += step) p.clear[i].ptr[x] = 0u;
}

inline cudaError_t launch_prompt_begin(PromptBeginParams& bp, const int32_t* lens_host, int batch, cudaStream_t st, int* n_launched) {
    unsigned long long most = kPbLens;
    for (const auto& c : bp.clear) most = std::max(most, c.words);
    const unsigned blocks = (unsigned)std::min<unsigned long long>(148, (most + kPbThreads - 1) / kPbThreads);
    *n_launched = 0;
    for (bp.first = 0; bp.first < batch; bp.first += kPbLens) {
        bp.n = std::min(kPbLens, batch - bp.first);
        std::memcpy(bp.lens, lens_host + bp.first, sizeof(int32_t) * (size_t)bp.n);
        prompt_begin_kernel<<<blocks, kPbThreads, 0, st>>>(bp);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        ++*n_launched;
    }
    return cudaSuccess;
}

// Host side. Returns CORM_ERR_UNSUPPORTED when the launch does not fit.
template <typename T, int D>
inline corm_status_t launch_prompt_cluster(const PromptParams& p, int G, int max_p, int sm_count, cudaStream_t st) {
    PromptClusterParams pp{};
    pp.p = p;
    while ((1 << pp.log2g) < G) ++pp.log2g;
    pp.rows8 = (p.w * G + 7) / 8 * 8;
    const int n_words = std::max(1, (max_p + 31) / 32);
    // As many blocks per unit as make the launch at least five waves of resident blocks: fewer leave the machine
    // to the longest units, more pay each block's fixed chain of round trips more often. us per pass with 1 / 2 / 4 / 8:
    // 1024 units x 3250 keys 969-1353 (with the slab's stride) / 956-1033 / 1073 / 1365, 128 units x 8192 keys (G 4) 2152 / 1281 / 811 / 752, 32 units x
    // 4096 keys 350 / 192 / 120 / 93.
    int cs = 1;
    while (cs < kPcMaxCluster && cs * 2 <= n_words && (long long)p.U * cs < 1500ll * sm_count / 148) cs *= 2;
    const PcSmem lay = pc_smem_layout<T, D>(pp.rows8);
    if (lay.total > 227 * 1024) return CORM_ERR_UNSUPPORTED;
    auto kern = prompt_cluster_kernel<T, D>;
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), (size_t)lay.total);
    if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)p.U, (unsigned)cs);
        cfg.blockDim = dim3(kPcThreads);
        cfg.dynamicSmemBytes = (size_t)lay.total;
        cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1;
        attr[0].val.clusterDim.y = (unsigned)cs;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        e = cudaLaunchKernelEx(&cfg, kern, pp);
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    if (e != cudaSuccess) { std::fprintf(stderr, "corm: prompt launch: %s\n", cudaGetErrorString(e)); return CORM_ERR_CUDA; }
    return CORM_OK;
}

}  // namespace corm
