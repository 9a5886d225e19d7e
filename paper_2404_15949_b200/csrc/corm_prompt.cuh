// Prompt-end pass: one launch, a thread-block cluster per unit (sequence x kv head), any dtype, head_dim and group.
//
// The min(P, w) recorded queries of the unit's G heads are R = w G "rows"; every row needs the log-sum-exp of its causal
// attention row (Eq. 2) before any verdict (Definition 3.1) can be taken. The cluster's blocks share the unit's keys
// (whole 32-key words each) and go through
//   A. logits of every row against the block's keys, summed as exp(s) per row (fp64, no running maximum: |s| below 650
//      cannot overflow);
//   -- the blocks exchange their sums through distributed shared memory: one threshold per row
//      (a unit with larger logits, or with bounds too wide to be of use, does A and B over in fp64: pc_fp64_rows)
//   B. verdicts of the block's keys for every row -> verdict registers;
//   -- the blocks exchange their counts of surviving keys
//   C. every block gathers its own survivors (K, V rows, registers, positions) to their place in token order.
// Keys stream through a ring of shared-memory buffers of 128 keys (asynchronous copies); a block whose keys fit the ring
// reads K once, otherwise later passes find it in L2 (a unit's K is a few MB and only as many units are in flight as fit the
// machine).
//
// bf16: both contractions run on the tensor cores (units of many rows: on tcgen05, corm_prompt_tc.cuh). Phase A needs fp64-grade logits: operands cut into exact pieces
// (corm_mma.cuh), 7 mma.m16n8k16 per 16 channels for 16 keys x 8 rows; the rows' pieces lie on chip for 32 rows at a time,
// and a warp's tile of keys is cut once for 16 of them. Phase B only has to place a logit on one side of its threshold: one
// plain mma per 16 channels, whose rounding is at most 2^-23 per term; the few logits inside that bound are formed again in
// fp64 by the whole warp (counted in corm_stats_t.near_threshold). If such a logit falls within the error of phase A's
// log-sum-exp itself, it is left open and the row is marked; after phase B the cluster forms the marked rows' log-sum-exps
// in fp64 and decides what was left open (about one row in 10^4..10^5). So every verdict is the fp64 one.
// fp32: fp64 arithmetic on the CUDA cores, lane = key, 4 rows at a time; only ties (1e-13) go to the exact rows, whose
// sums keep the largest logit apart, so that a query at position 1 stays exactly on its threshold.
//
// What bounds it: for windows of a few queries HBM and the latency of the gather (K once, the survivors' V in, K and V
// out); for more rows, below those that tc_takes gives to tcgen05, the tensor pipe's mma.sync rate in phase A (R P d
// multiply-adds, seven times).
// Measured, us per pass: a two-launch pass (fp64 logits on the CUDA cores; one block per unit gathering; for fp32 or 64
// channels one block per unit for everything) -> a first cluster pass (a warp per octet of rows, every warp cutting every
// key; marked rows a key at a time) -> now on mma.sync (of which products without a zeroed addend, fragment addresses from one lane
// constant and exponentials without a range check, which the limit on the logits makes needless: 1755 -> 1699 at w 128):
//   1024 units x 3250 keys, G 1, w 8    1597 -> 1036 ->  840    128 units x 3390 keys, G 1, w 256    5341 -> 1709 -> 1582 (tcgen05: 905)
//   128 units x 8192 keys, G 4, w 8     1821 ->  769 ->  598    32 units x 8192 keys, G 4, w 128     6736 -> 2206 -> 1699 (tcgen05: 1045)
//   32 units x 32768 keys, G 4, w 16    4618 -> 2375 -> 1049    32 units x 4096 keys, G 1, w 8        259 ->   65 ->   60
//   fp32: 20 units x 1300 keys, G 2     2787 ->  103            64 channels: 128 units x 2000, G 4  11037 ->  273 ->  238
#pragma once

#include "corm_fast.cuh"
#include "corm_prompt_rows.cuh"
#include "corm_prompt_tc.cuh"

namespace corm {

constexpr int kTcMinRows = 96;                  // rows of a unit from which phases A and B may run on tcgen05
// Bound of a logit's error, times the prompt's keys, beyond which a unit does both phases in fp64: so many verdicts would be
// left open that most rows are formed apart. us per pass, tensor cores / fp64, one key channel 256 and 1024 times the others:
// mma.sync 32 units x 32768 keys, G 4, w 16, 6240 / 4210 and 13440 / 4210; 1024 x 3250, w 8, 1570 / 3100 and 3070 / 3180; tcgen05
// 32 x 8192, G 4, w 128, 10500 / 7360 and 24650 / 7360; 128 x 3390, w 256, 3520 / 6650 and 10360 / 6650; 32 x 2000, w 256, 650 /
// 950 and 1750 / 950; 16 x 8192, w 128, 1450 / 1820 and 3860 / 1820 (fp64 inside the mma.sync launch: 8140, 6770, 1060 and 1810).
constexpr double kPcReachKeys = 1.2;

struct PromptClusterParams {
    PromptParams p;
    int32_t log2g;
    int32_t rows8;           // w G rounded up to a multiple of 8
};

template <typename T, int D>
__host__ __device__ inline PcSmem pc_smem_layout(int rows8) {
    PcSmem s{};
    int off = 0;
    auto take = [&](int bytes) { int at = off; off = (off + bytes + 127) / 128 * 128; return at; };
    s.ring = take(pc_bufs<T, D>(rows8) * kPcKeys * D * Elem<T>::kBytes);
    s.zs = take((rows8 > 64 ? rows8 : 64) * 8);
    s.thr = take(rows8 * 8);
    s.n1 = take(rows8 * 4);
    s.qe = take(rows8 * 4);
    s.flags = take((rows8 + 31) / 32 * 4);
    s.words = take(Elem<T>::kBytes == 4 ? kPcKeys * 4 : 0);
    s.list = take(kPcWarps * 32);               // gather: the kept lanes of a warp's word
    s.stage = take(Elem<T>::kBytes == 4 ? kPcWarps * 4 * D * 8 : 0);
    // bf16: pieces of a group's octets (three of 256 bytes per 16 channels), or raw values of twice as many (one)
    const int octets = rows8 / 8, even = octets == 1 ? 1 : (octets + 1) / 2 * 2;
    const int fa = (even < kPcGroup ? even : kPcGroup) * (D / 16) * 3 * 256, fb = (octets < kPcGroupB ? octets : kPcGroupB) * (D / 16) * 256;
    s.frag = take(Elem<T>::kBytes == 2 ? (fa > fb ? fa : fb) : 0);
    s.misc = take((int)sizeof(PcMisc));
    s.total = off;
    return s;
}

// byte offset of 16-byte chunk c of row r inside a ring buffer (rows of D elements, chunk index XOR row mod 8)
template <typename T, int D> __device__ __forceinline__ int pc_offset(int r, int c) { return r * (D * Elem<T>::kBytes) + ((c ^ (r & 7)) << 4); }

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

// The marked rows, exactly, by all blocks of the cluster: log-sum-exp in fp64 with a running maximum, then the verdicts that
// phase B left open (misc->open, or every key where those did not fit). Verdicts that phase B was sure of hold
// for the exact threshold too, so adding marks is enough. Rare, but a launch is as long as its longest unit: with a key at a
// time per warp and a second pass over the keys for the verdicts this took 714 us of 1592 on 32768-key prompts.
template <typename T, int D>
__device__ __noinline__ void pc_exact_rows(const PromptParams& p, const PcRows& R, const T* Qu, const T* Ku, int k_begin, int k_end,
                                           const uint32_t* flags, uint32_t* words_g, PcMisc* misc, int cs) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, sub = lane & 3;
    const uint32_t mz_addr = smem_addr(misc->mz);
    auto row_of = [&](int j) -> const T* { return Ku + (size_t)j * D; };
    const int n_open = misc->n_open > kPcOpenCap ? -1 : misc->n_open;
    for (int r = 0; r < R.rows; ++r) {
        if (!((flags[r >> 5] >> (r & 31)) & 1u)) continue;
        const int qpos = R.pos(r);
        if (!qpos) continue;
        const T* qr = R.q<T, D>(Qu, r);
        const int end = min(k_end, qpos);                     // causal row: keys 1..position of the query
        double m, Z;
        warp_exact_lse<T, D>(qr, row_of, k_begin + warp * 16, end, kPcWarps * 16, m, Z);
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
        QuadRow<T, D> q;
        q.load(qr, sub);
        const int n = n_open < 0 ? max(0, end - k_begin) : n_open;
        for (int i0 = warp * 8; i0 < n; i0 += kPcWarps * 8) {  // eight keys per warp, the same sums as above
            const int i = i0 + (lane >> 2);
            const bool on = i < n && (n_open < 0 || misc->open[i].x == r);
            const int j = on ? (n_open < 0 ? k_begin + i : misc->open[i].y) : k_begin;
            const T* const rows[1] = {row_of(j)};
            double s[1];
            quad_exact_dots<T, D, 1>(q, rows, sub, s);
            if (on && sub == 0 && s[0] * inv_root_dim(D) >= thr) words_g[j] = pc_join(p.w, __ldcg(words_g + j), pc_mark(p.w, R.rho(r), qpos));
        }
        cluster_sync();                                       // everybody has read mz; the marks of this row are written
    }
}

// Units whose logits are too large for plain sums of exponentials (650 and more), whose elements the pieces cannot hold, or
// whose error bounds are too wide to be of use: both phases in fp64 on the CUDA cores, with running maxima. A warp owns units
// of four rows (the queries widened in shared memory), a lane one or two keys; warps share rows by groups of 32 keys where
// there are fewer than eight row units. On return the thresholds and the scratch registers are there; rows are marked, and
// their keys listed, for ties only. key_buf: 128 rows of keys, q_stage: room for `room` units of doubles per warp (a warp with no
// more than that widens its rows once; else for every chunk of keys, which a block on tcgen05, with little L1, pays for: 16 units x
// 8192 keys, 128 rows, 2007 -> 1817 us), words: 128 registers.
template <typename T, int D>
__device__ __noinline__ void pc_fp64_rows(const PromptParams& p, const PcRows& R, const T* Qu, const T* Ku, int k_begin, int n_keys, unsigned char* key_buf,
                                          double* q_stage, int room, double* zs, double* thr_sm, uint32_t* words, uint32_t* words_g, uint32_t* flags, PcMisc* misc, int cs) {
    constexpr int kRow = D * Elem<T>::kBytes, kChunks = kRow / 16, kEl = 16 / Elem<T>::kBytes, kSubs = kPcKeys / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nc = (n_keys + kPcKeys - 1) / kPcKeys;
    const int n_ru = (R.rows + 3) / 4;
    int slots = 1;                                            // warps side by side over the row units (a power of two)
    while (slots < n_ru && slots < kPcWarps) slots *= 2;
    const int groups = min(kPcWarps / slots, kSubs), my_ru = warp % slots, my_kg = warp / slots;
    const bool works = my_ru < n_ru && my_kg < groups;
    double* q = q_stage + warp * room * 4 * D;
    const bool kept = (n_ru + slots - 1) / slots <= room;
    double* const ms = groups > 1 ? zs + 32 : thr_sm;         // running maxima next to the sums (fewer than 32 rows x groups)
    auto load = [&](int c) {
        __syncthreads();                                      // everybody is done with the chunk before
        const unsigned char* src = reinterpret_cast<const unsigned char*>(Ku + (size_t)(k_begin + c * kPcKeys) * D);
        const int valid = n_keys - c * kPcKeys;
#pragma unroll 8
        for (int x = tid; x < kPcKeys * kChunks; x += kPcThreads) {
            const int r = x / kChunks;
            *reinterpret_cast<uint4*>(key_buf + pc_offset<T, D>(r, x % kChunks)) = r < valid ? __ldg(reinterpret_cast<const uint4*>(src) + x) : make_uint4(0, 0, 0, 0);
        }
        __syncthreads();
    };
    auto stage = [&](int ru, bool first) {                    // unit ru's rows in q
        q = q_stage + (warp * room + (kept ? ru / slots : 0)) * 4 * D;
        if (kept && !first) return;
        __syncwarp();
        for (int x = lane; x < 4 * D; x += 32) {
            const int r = ru * 4 + x / D;
            q[x] = R.pos(r) ? (double)Elem<T>::load(R.template q<T, D>(Qu, r) + x % D) : 0.0;
        }
        __syncwarp();
    };
    // logits of the staged rows against the lane's keys of one group of 32, or of two
    auto logits = [&](int sub, bool two, double (&s)[2][4]) {
        const int r0 = sub * 32 + lane, r1 = two ? r0 + groups * 32 : r0;
#pragma unroll
        for (int x = 0; x < 4; ++x) s[0][x] = s[1][x] = 0.0;
#pragma unroll 2
        for (int ch = 0; ch < kChunks; ++ch) {
            double k[2][kEl];
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                const uint4 raw = *reinterpret_cast<const uint4*>(key_buf + pc_offset<T, D>(y ? r1 : r0, ch));
                if constexpr (kEl == 8) {
                    unpack8_to_double(raw, k[y]);
                } else {
                    k[y][0] = (double)__uint_as_float(raw.x); k[y][1] = (double)__uint_as_float(raw.y);
                    k[y][2] = (double)__uint_as_float(raw.z); k[y][3] = (double)__uint_as_float(raw.w);
                }
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int e = 0; e < kEl; e += 2) {
                    const double2 a = *reinterpret_cast<const double2*>(q + x * D + ch * kEl + e);
#pragma unroll
                    for (int y = 0; y < 2; ++y) { s[y][x] = fma(a.x, k[y][e], s[y][x]); s[y][x] = fma(a.y, k[y][e + 1], s[y][x]); }
                }
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) { s[0][x] *= inv_root_dim(D); s[1][x] *= inv_root_dim(D); }
    };
    auto join = [](double& m, double& z, double mo, double zo) {          // (log-)sums of exponentials
        const double mn = fmax(m, mo);
        z = z * exp_nonpos(m - mn) + zo * exp_nonpos(mo - mn);
        m = mn;
    };

    // A. per row: largest logit and sum of exponentials below it
    for (int i = tid; i < (groups > 1 ? 32 : n_ru * 4); i += kPcThreads) { zs[i] = 0.0; ms[i] = -INFINITY; }
    for (int c = 0; c < nc; ++c) {
        load(c);
        const int n_valid = min(kPcKeys, n_keys - c * kPcKeys);
        if (!works) continue;
        for (int ru = my_ru; ru < n_ru; ru += slots) {
            stage(ru, c == 0);
            double m[4], z[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) { m[x] = -INFINITY; z[x] = 0.0; }
            for (int sub = my_kg; sub < kSubs && sub * 32 < n_valid; sub += 2 * groups) {
                const bool two = sub + groups < kSubs && (sub + groups) * 32 < n_valid;
                double s[2][4];
                logits(sub, two, s);
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    const int at = (sub + y * groups) * 32 + lane, j = k_begin + c * kPcKeys + at;
                    if (y && !two) continue;
#pragma unroll
                    for (int x = 0; x < 4; ++x)
                        if (at < n_valid && j < R.pos(ru * 4 + x)) join(m[x], z[x], s[y][x], 1.0);      // causal row
                }
            }
#pragma unroll
            for (int x = 0; x < 4; ++x) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) join(m[x], z[x], __shfl_xor_sync(0xffffffffu, m[x], o), __shfl_xor_sync(0xffffffffu, z[x], o));
                if (lane == 0) {                              // the warp's own place
                    const int at = my_kg * (n_ru * 4) + ru * 4 + x;
                    join(m[x], z[x], ms[at], zs[at]);
                    ms[at] = m[x]; zs[at] = z[x];
                }
            }
        }
    }
    __syncthreads();
    if (groups > 1) {                                         // the groups of this block
        double m = -INFINITY, z = 0.0;
        if (tid < n_ru * 4)
            for (int x = 0; x < groups; ++x) join(m, z, ms[x * (n_ru * 4) + tid], zs[x * (n_ru * 4) + tid]);
        __syncthreads();
        if (tid < n_ru * 4) { zs[tid] = z; thr_sm[tid] = m; }
    }
    cluster_sync();
    constexpr int kPer = 2048 / kPcThreads;                   // rows per thread (256 queries of eight heads at most)
    double t[kPer];
#pragma unroll
    for (int y = 0; y < kPer; ++y) {
        const int r = tid + y * kPcThreads;
        double m = -INFINITY, z = 0.0;
        if (r < R.rows)
            for (int x = 0; x < cs; ++x) join(m, z, ld_peer_f64(map_rank(smem_addr(thr_sm + r), x)), ld_peer_f64(map_rank(smem_addr(zs + r), x)));
        t[y] = r < R.rows && R.pos(r) ? m + log(z) + p.log_alpha - log((double)R.pos(r)) : INFINITY;
    }
    cluster_sync();                                           // everybody has read everybody's sums
#pragma unroll
    for (int y = 0; y < kPer; ++y)
        if (tid + y * kPcThreads < R.rows) thr_sm[tid + y * kPcThreads] = t[y];

    // B. verdicts
    for (int c = 0; c < nc; ++c) {
        load(c);                                              // (the thresholds are there behind its barriers)
        if (tid < kPcKeys) words[tid] = 0u;
        __syncthreads();
        const int n_valid = min(kPcKeys, n_keys - c * kPcKeys);
        if (works)
            for (int ru = my_ru; ru < n_ru; ru += slots) {
                stage(ru, false);
                for (int sub = my_kg; sub < kSubs && sub * 32 < n_valid; sub += 2 * groups) {
                    const bool two = sub + groups < kSubs && (sub + groups) * 32 < n_valid;
                    double s[2][4];
                    logits(sub, two, s);
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        const int at = (sub + y * groups) * 32 + lane, j = k_begin + c * kPcKeys + at;
                        if ((y && !two) || at >= n_valid) continue;
                        uint32_t mark = 0u;
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int row = ru * 4 + x, qpos = R.pos(row);
                            if (j >= qpos) continue;
                            const double th = thr_sm[row], margin = s[y][x] - th, e = th > -INFINITY ? 1e-13 * (1.0 + fabs(th)) : 0.0;
                            if (margin > e) mark = pc_join(p.w, mark, pc_mark(p.w, R.rho(row), qpos));
                            else if (margin >= -e) pc_leave_open(flags, misc, row, j);
                        }
                        if (mark) {
                            if (p.w <= 32) atomicOr(words + at, mark);
                            else atomicMax(words + at, mark);
                        }
                    }
                }
            }
        __syncthreads();
        if (tid < n_valid) words_g[k_begin + c * kPcKeys + tid] = words[tid];
    }
    __syncthreads();
}

// Raw values of 8 rows in the B operand's layout (row n = lane / 4); zeros for rows that do not exist.
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

// The pieces of 8 rows (b1 and b2 as one 16-byte word per lane and 16 channels, b3 as one of 8), and the rows' norms for
// the error bounds. Returns false if a row leaves the safe range.
template <int D>
__device__ __noinline__ bool pc_store_pieces(const PcRows& R, const bf16_t* Qu, int octet, int lane, uint4* f12, uint2* f3, float* n1_sm, float* qe_sm) {
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
    for (int kk = 0; kk < D / 16; ++kk) {
        uint32_t b[2][3];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float a[2] = {__uint_as_float(raw[kk][h] << 16), __uint_as_float(raw[kk][h] & 0xffff0000u)}, x1[2], x2[2], x3[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                split_query(a[e], c, x1[e], x2[e], x3[e]);
                n1 += fabsf(a[e]); n2 += fabsf(x2[e]); n3 += fabsf(x3[e]);
            }
            b[h][0] = (__float_as_uint(x1[0]) >> 16) | (__float_as_uint(x1[1]) & 0xffff0000u);   // exact: bf16 numbers
            b[h][1] = (__float_as_uint(x2[0]) >> 16) | (__float_as_uint(x2[1]) & 0xffff0000u);
            b[h][2] = (__float_as_uint(x3[0]) >> 16) | (__float_as_uint(x3[1]) & 0xffff0000u);
        }
        f12[kk * 32 + lane] = make_uint4(b[0][0], b[1][0], b[0][1], b[1][1]);
        f3[kk * 32 + lane] = make_uint2(b[0][2], b[1][2]);
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        n1 += __shfl_xor_sync(0xffffffffu, n1, o);
        n2 += __shfl_xor_sync(0xffffffffu, n2, o);
        n3 += __shfl_xor_sync(0xffffffffu, n3, o);
    }
    if ((lane & 3) == 0 && 8 * octet < (R.rows + 7) / 8 * 8) {
        n1_sm[8 * octet + (lane >> 2)] = n1 * 1.0001f;
        qe_sm[8 * octet + (lane >> 2)] = split_error(n1, n2, n3);
    }
    return ok;
}

// exp(s) of 16 keys against N octets of rows, added to z[octet][row pair's two]; `last`: the tile may hold keys that a row
// does not see or that do not exist (qpos: the rows' positions). Returns the largest high word of |s|.
template <int D, int N>
__device__ __forceinline__ uint32_t pc_tile_sums(uint32_t tile, uint32_t klane, SplitGrid g, int lane, const uint4* f12, const uint2* f3, int j0, int k_end, bool last,
                                                 const PcRows& R, int row0, double (*z)[2]) {
    float hi[N][4], mid[N][4], lo[N][4];
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
        uint32_t a[4], k1[4], k2[4], r2[4];
        ldmatrix_x4(a, tile + (klane ^ (kk << 5)));
        split_key(a, g, k1, k2, r2);
#pragma unroll
        for (int o = 0; o < N; ++o) {
            const uint4 b = f12[(o * (D / 16) + kk) * 32 + lane];
            const uint2 b3 = f3[(o * (D / 16) + kk) * 32 + lane];
            float t[4];
            if (kk == 0) {
                mma16816_zero(hi[o], k1, b.x, b.y);
                mma16816_zero(mid[o], k1, b.z, b.w);
            } else {
                mma16816(hi[o], k1, b.x, b.y);
                mma16816(mid[o], k1, b.z, b.w);
            }
            mma16816_zero(t, k2, b.z, b.w);
            mma16816(t, r2, b.x, b.y);
            mma16816(mid[o], k2, b.x, b.y);
            mma16816(t, r2, b.z, b.w);
            mma16816(t, k1, b3.x, b3.y);
#pragma unroll
            for (int x = 0; x < 4; ++x) lo[o][x] = kk == 0 ? t[x] : lo[o][x] + t[x];
        }
    }
    uint32_t top = 0u;
    const double inv_root_d = inv_root_dim(D);
#pragma unroll
    for (int o = 0; o < N; ++o)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const double s = (((double)hi[o][x] + (double)mid[o][x]) + (double)lo[o][x]) * inv_root_d;
            double e = exp_reduced(s);                        // (any s beyond kPcLogitLimit sends the unit through pc_fp64_rows)
            uint32_t h = (uint32_t)__double2hiint(s) & 0x7fffffffu;
            if (last) {                                       // causal row: keys 1..position of the query
                const int j = j0 + (lane >> 2) + (x >> 1) * 8;
                if (j >= k_end || j >= R.pos(row0 + o * 8 + 2 * (lane & 3) + (x & 1))) { e = 0.0; h = 0u; }
            }
            top = max(top, h);
            z[o][x & 1] += e;
        }
    return top;
}

// largest magnitude (bf16 bits) of a 16-key tile, by the warp that works on it
template <int D>
__device__ __forceinline__ uint32_t pc_tile_amax(const unsigned char* tile, int lane) {
    uint32_t m = 0u;
#pragma unroll
    for (int x = 0; x < D / 16; ++x) {
        const uint4 v = *reinterpret_cast<const uint4*>(tile + (x * 32 + lane) * 16);
        m = max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(m, v.x), v.y), v.z), v.w);
    }
    return __reduce_max_sync(0xffffffffu, max(m & 0xffffu, m >> 16));
}

// Verdicts that the bounds leave open, by a whole warp: bit x of `open` = key j0 + lane / 4 + 8 (x / 2) against row
// row0 + 2 (lane % 4) + x % 2. Adds to the lane's marks what is sure; rows whose threshold is too close are flagged.
template <typename T, int D>
__device__ __noinline__ void pc_open_verdicts(const PromptParams& p, const PcRows& R, const T* Qu, const T* Ku, int j0, int row0, uint32_t open,
                                              const double* thr_sm, const float* qe_sm, double eps_unit, uint32_t* flags, PcMisc* misc, uint32_t (&mark)[2]) {
    const int lane = threadIdx.x & 31;
    int n_near = 0;
    for (int x = 0; x < 4; ++x) {
        uint32_t who = __ballot_sync(0xffffffffu, (open >> x) & 1u);
        n_near += __popc(who);
        while (who) {
            const int src = __ffs(who) - 1;
            who &= who - 1u;
            const int j = j0 + (src >> 2) + (x >> 1) * 8, row = row0 + 2 * (src & 3) + (x & 1);
            const double s = warp_exact_dot<T, D>(R.q<T, D>(Qu, row), Ku + (size_t)j * D, lane) * inv_root_dim(D);
            const double th = thr_sm[row], e = eps_unit * (double)qe_sm[row] + 1e-13 * (1.0 + fabs(th));
            if (lane == src && s - th > e) mark[x >> 1] = pc_join(p.w, mark[x >> 1], pc_mark(p.w, R.rho(row), R.pos(row)));
            if (lane == 0 && fabs(s - th) <= e) pc_leave_open(flags, misc, row, j);   // to the exact rows
        }
    }
    if (lane == 0) atomicAdd(p.counters + CNT_NEAR, (unsigned long long)n_near);
}

// kTc: phases A and B on tcgen05 (corm_prompt_tc.cuh)
template <typename T, int D, bool kTc>
__global__ void __launch_bounds__(kTc ? kTcThreads : kPcThreads, !kTc && D * Elem<T>::kBytes <= 256 ? 2 : 1)
prompt_cluster_kernel(const __grid_constant__ PromptClusterParams pp) {
    extern __shared__ __align__(128) unsigned char smem[];
    const PromptParams& p = pp.p;
    constexpr bool kBf16 = Elem<T>::kBytes == 2;
    constexpr int kRow = D * Elem<T>::kBytes, kChunks = kRow / 16;
    constexpr int kSubs = kPcKeys / 32;                       // fp32: units of 32 keys per buffer
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
    PcSmem lay;
    if constexpr (kTc) lay = tc_smem_layout<D>(pp.rows8); else lay = pc_smem_layout<T, D>(pp.rows8);
    const int n_buf = pc_bufs<T, D>(pp.rows8);
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
    const bool resident = nc <= n_buf;                        // the block's keys stay on chip for all passes over them
    const T* Ku = reinterpret_cast<const T*>(p.k_prompt) + (size_t)u * p.p_max * D;
    const T* Vu = reinterpret_cast<const T*>(p.v_prompt) + (size_t)u * p.p_max * D;
    const T* Qu = reinterpret_cast<const T*>(p.q_last) + ((size_t)u << pp.log2g) * w * D;
    uint32_t* words_g = reinterpret_cast<uint32_t*>(p.stash) + (size_t)u * p.C;      // scratch registers of this unit
    const double inv_root_d = inv_root_dim(D), root_d = D == 128 ? 11.313708498984760390 : 8.0;
    const uint32_t ring = smem_addr(smem + lay.ring);

    // Passes over the block's keys take numbered steps, step s = chunk s % nc in ring buffer s % n_buf (a resident block
    // loads every chunk once). Loads run n_buf - 1 steps ahead, `end` steps in all.
    auto issue = [&](int step, int end) {
        if (step < end) {
            const int c = step % nc;
            const uint32_t dst = ring + (step % n_buf) * (kPcKeys * kRow);
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
    auto start = [&](int end) { for (int i = 0; i < n_buf - 1; ++i) issue(i, end); };
    // waits for the step's chunk and starts the load n_buf - 1 steps on; returns the chunk's buffer
    auto arrive = [&](int step, int end) -> const unsigned char* {
        if (n_buf == 3) cp_async_wait<1>(); else cp_async_wait<0>();
        __syncthreads();                                      // the chunk is in; everybody is done with the buffer that is filled next
        issue(step + n_buf - 1, end);
        return smem + lay.ring + (resident ? step % nc : step % n_buf) * (kPcKeys * kRow);
    };
    const int n_oct = pp.rows8 / 8;
    const int n_grp = kBf16 ? (n_oct + kPcGroup - 1) / kPcGroup : 1;                 // passes of phase A
    const int end_a = resident ? nc : n_grp * nc;
    if (!kTc) start(end_a);
    for (int i = tid; i < (pp.rows8 + 31) / 32; i += kPcThreads) flags[i] = 0u;
    if (tid == 0) { misc->bad = 0; misc->amax = 0u; misc->fail = 0; misc->n_open = 0; }

    // ---- A. sums of exp(s) per row ----
    bool bad = false;
    // fp32: warps own units of four rows where there are at least as many, otherwise they share them by key units
    const int n_ru = (R.rows + 3) / 4;
    int ru_slots = 1;                                         // warps side by side over the row units (a power of two)
    while (ru_slots < n_ru && ru_slots < kPcWarps) ru_slots *= 2;
    const int key_groups = min(kPcWarps / ru_slots, kSubs);
    const int my_ru = warp % ru_slots, my_kg = warp / ru_slots;
    const bool works = my_ru < n_ru && my_kg < key_groups;
    const bool keep_rows = n_ru <= ru_slots;                  // a warp has one row unit at most: it stays staged
    double* qst = reinterpret_cast<double*>(smem + lay.stage) + warp * 4 * D;        // fp32: the rows as doubles
    auto stage_rows = [&](int ru) {
        __syncwarp();
        for (int x = lane; x < 4 * D; x += 32) {
            const int r = ru * 4 + x / D;
            qst[x] = R.pos(r) ? (double)Elem<T>::load(R.q<T, D>(Qu, r) + x % D) : 0.0;
        }
        __syncwarp();
    };
    auto dot4 = [&](const unsigned char* buf, int kr, double (&acc)[4]) {           // the staged rows against key kr of the buffer
#pragma unroll
        for (int x = 0; x < 4; ++x) acc[x] = 0.0;
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
    };
    uint4* f12 = reinterpret_cast<uint4*>(smem + lay.frag);
    // a lane's offset for fragment loads inside a tile: chunk 2 kk of its row is one exclusive-or with kk << 5 away
    const uint32_t klane = (lane & 15) * kRow + (((lane >> 4) ^ (lane & 7)) << 4);
    TcMisc* tc = reinterpret_cast<TcMisc*>(smem + lay.tc);
    TcBlock block{R, reinterpret_cast<const bf16_t*>(Qu), reinterpret_cast<const bf16_t*>(Ku), k_begin, k_end, n_keys, smem + lay.ring, tc, 0u, 0, false};
    if constexpr (kTc) {
        if (tid == 0) {
            mbar_init(smem_addr(tc->bar), 1);
            mbar_init(smem_addr(tc->bar + 1), 1);
            mbar_init(smem_addr(tc->full), kPcWarps);
            mbar_init(smem_addr(tc->full + 1), kPcWarps);
            fence_mbar_init();
        }
        if (tid < 16) tc->exp16[tid] = TcExp<D>::entry(tid);
        if (warp == 0) tc_alloc(smem_addr(&tc->tmem));
        tc_before_sync();
        __syncthreads();
        tc_after_sync();
        block.tmem = tc->tmem;
        if (warp == kPcWarps) {                               // its work is done with phase A's products (barriers don't count it then)
            tc_issue_a<D>(block);
            return;
        }
        bad = !tc_phase_a<D>(block, zs, n1_sm, qe_sm, &misc->amax) || (smem_addr(smem) & 1023u);     // (the swizzle's alignment; never expected)
    } else if constexpr (kBf16) {
        // A group of four octets of rows at a time: its pieces are made once and stay on chip while the block's keys pass;
        // a warp takes one tile of every chunk, cuts it into pieces once per two octets and keeps its rows' sums in
        // registers to the end of the pass.
        uint32_t top = 0u;
        for (int grp = 0; grp < n_grp; ++grp) {
            const int oct0 = grp * kPcGroup, cnt = min(kPcGroup, n_oct - oct0), n_even = n_oct == 1 ? 1 : (cnt + 1) / 2 * 2;
            uint2* f3 = reinterpret_cast<uint2*>(f12 + (n_oct == 1 ? 1 : min((n_oct + 1) / 2 * 2, kPcGroup)) * (D / 16) * 32);
            if (grp) __syncthreads();                         // everybody is done with the group before
            if (warp < n_even)
                bad |= !pc_store_pieces<D>(R, Qu, oct0 + warp, lane, f12 + warp * (D / 16) * 32, f3 + warp * (D / 16) * 32, n1_sm, qe_sm);
            double z[kPcGroup][2];
#pragma unroll
            for (int o = 0; o < kPcGroup; ++o) z[o][0] = z[o][1] = 0.0;
            if (nc == 0) __syncthreads();
            for (int c = 0; c < nc; ++c) {
                const unsigned char* buf = arrive(grp * nc + c, end_a);
                const int n_valid = min(kPcKeys, n_keys - c * kPcKeys), j0 = k_begin + c * kPcKeys + warp * 16;
                if (warp * 16 >= n_valid) continue;
                const uint32_t am = pc_tile_amax<D>(buf + warp * 16 * kRow, lane);
                if (grp == 0 && lane == 0) atomicMax(&misc->amax, am);
                const SplitGrid g = split_grid(am);
                const uint32_t tile = smem_addr(buf) + warp * 16 * kRow;
                const bool last = j0 + 16 > k_end || j0 + 16 > P - w + 1;
                if (n_oct == 1) {
                    top = max(top, pc_tile_sums<D, 1>(tile, klane, g, lane, f12, f3, j0, k_end, last, R, 0, z));
                } else {
                    top = max(top, pc_tile_sums<D, 2>(tile, klane, g, lane, f12, f3, j0, k_end, last, R, oct0 * 8, z));
                    if (cnt > 2)
                        top = max(top, pc_tile_sums<D, 2>(tile, klane, g, lane, f12 + 2 * (D / 16) * 32, f3 + 2 * (D / 16) * 32, j0, k_end, last, R, oct0 * 8 + 16, z + 2));
                }
            }
#pragma unroll
            for (int o = 0; o < kPcGroup; ++o) {
#pragma unroll
                for (int x = 4; x < 32; x <<= 1) { z[o][0] += __shfl_xor_sync(0xffffffffu, z[o][0], x); z[o][1] += __shfl_xor_sync(0xffffffffu, z[o][1], x); }
                if (lane < 4) { misc->zw[warp][o * 8 + 2 * lane] = z[o][0]; misc->zw[warp][o * 8 + 2 * lane + 1] = z[o][1]; }
            }
            __syncthreads();
            if (tid < cnt * 8) {
                double t = 0.0;
                for (int x = 0; x < kPcWarps; ++x) t += misc->zw[x][tid];
                zs[oct0 * 8 + tid] = t;
            }
        }
        bad |= top >= (uint32_t)__double2hiint(kPcLogitLimit);
    } else {
        double z[4] = {0.0, 0.0, 0.0, 0.0};
        for (int i = tid; i < max(pp.rows8, 64); i += kPcThreads) zs[i] = 0.0;
        auto fold = [&](int ru) {                             // the warp's lanes -> its slots of zs
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const double t = warp_sum(z[x]);
                if (lane == 0) zs[my_kg * (n_ru * 4) + ru * 4 + x] += t;
                z[x] = 0.0;
            }
        };
        bool have = false;
        for (int c = 0; c < nc; ++c) {
            const unsigned char* buf = arrive(c, end_a);
            const int n_valid = min(kPcKeys, n_keys - c * kPcKeys);
            if (works)
                for (int ru = my_ru; ru < n_ru; ru += ru_slots) {
                    if (!keep_rows || !have) stage_rows(ru);
                    have = true;
                    int qpos[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) qpos[x] = R.pos(ru * 4 + x);
                    for (int sub = my_kg; sub < kSubs && sub * 32 < n_valid; sub += key_groups) {
                        double acc[4];
                        dot4(buf, sub * 32 + lane, acc);
                        const int j = k_begin + c * kPcKeys + sub * 32 + lane;
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const double s = acc[x] * inv_root_d;
                            const bool on = j < k_end && j < qpos[x];               // causal row: keys 1..position of the query
                            bad |= on && !(fabs(s) < kPcLogitLimit);
                            z[x] += on ? exp_reduced(s) : 0.0;
                        }
                    }
                    if (!keep_rows) fold(ru);
                }
        }
        __syncthreads();
        if (works && keep_rows) fold(my_ru);
    }
    if (bad) misc->bad = 1;
    __syncthreads();
    if (kBf16 && tid == 0 && misc->amax >= kSplitMaxBits) misc->bad = 1;
    if (!kBf16)
        for (int i = tid; i < n_ru * 4; i += kPcThreads)      // key groups of this block, in a fixed order
            for (int x = 1; x < key_groups; ++x) zs[i] += zs[x * (n_ru * 4) + i];
    cluster_sync();

    // ---- thresholds of Definition 3.1 in log form: s >= lse + ln(alpha) - ln(position of the query) ----
    int any_bad = 0;
    uint32_t amax_unit = 0u;
    for (int x = 0; x < cs; ++x) {
        any_bad |= (int)ld_peer_u32(map_rank(smem_addr(&misc->bad), x));
        amax_unit = max(amax_unit, ld_peer_u32(map_rank(smem_addr(&misc->amax), x)));
    }
    for (int r = tid; r < R.rows; r += kPcThreads) {
        const int qpos = R.pos(r);
        double Z = 0.0;
        for (int x = 0; x < cs; ++x) Z += ld_peer_f64(map_rank(smem_addr(zs + r), x));
        thr_sm[r] = qpos ? log(Z) + p.log_alpha - log((double)qpos) : INFINITY;
    }
    // error of a threshold per unit of qe (every logit of the row is off by at most this much, so its log-sum-exp is too)
    const double eps_unit = kBf16 ? p.bound_scale * (double)split_amax(amax_unit) * inv_root_d : 0.0;
    bool wide = any_bad != 0;                                 // the same in every block: unit and rows are
    if constexpr (kBf16)
        if (!wide)
            for (int r = tid; r < R.rows; r += kPcThreads) wide |= eps_unit * qe_sm[r] * (double)P > kPcReachKeys * p.bound_scale;
    wide = __syncthreads_or(wide);

    // ---- B. verdicts -> registers ----
    const int n_grp_b = kBf16 ? (n_oct + kPcGroupB - 1) / kPcGroupB : 1;
    const int end_b = resident || wide ? 0 : n_grp_b * nc;
    if (!kTc && !resident && !wide) start(end_b);
    if (wide) {
        cluster_sync();                                       // everybody has read everybody's sums of phase A
        constexpr int kBuf = kPcKeys * kRow;
        static_assert(kPcWarps * 4 * D * 8 <= kBuf, "the widened rows fit a ring buffer");
        pc_fp64_rows<T, D>(p, R, Qu, Ku, k_begin, n_keys, smem + lay.ring, reinterpret_cast<double*>(smem + lay.ring + kBuf), kTc ? kTcRowRoom : 1, zs, thr_sm,
                           kBf16 ? reinterpret_cast<uint32_t*>(f12) : words_sm, words_g, flags, misc, cs);
    } else if constexpr (kTc) {
        tc_phase_b<D>(p, block, thr_sm, n1_sm, qe_sm, eps_unit, words_g, flags, misc);
    } else if constexpr (kBf16) {
        uint2* fr = reinterpret_cast<uint2*>(f12);
        for (int grp = 0; grp < n_grp_b; ++grp) {
            const int oct0 = grp * kPcGroupB, cnt = min(kPcGroupB, n_oct - oct0);
            __syncthreads();                                  // thresholds are there; everybody is done with the group before
            if (warp < cnt) {
                uint32_t raw[D / 16][2];
                pc_load_raw<D>(R, Qu, oct0 + warp, lane, raw);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) fr[(warp * (D / 16) + kk) * 32 + lane] = make_uint2(raw[kk][0], raw[kk][1]);
            }
            if (tid < cnt * 8) {
                const int r = oct0 * 8 + tid;
                const float tf = r < R.rows ? (float)(thr_sm[r] * root_d) : INFINITY;
                misc->thr_f[tid] = tf;
                // D roundings of 2^-23 on sums of at most A |q|_1 (a tenth of slack), the threshold's own rounding, and the
                // threshold's error
                misc->err_f[tid] = (float)p.bound_scale * ((float)D * 1.1f / 8388608.f * n1_sm[r]);
                misc->slack[tid] = (tf < 3e38f ? fabsf(tf) : 0.f) * 2.4e-7f + (float)(eps_unit * qe_sm[r] * root_d) * 1.01f;
            }
            if (nc == 0) __syncthreads();
            for (int c = 0; c < nc; ++c) {
                const unsigned char* buf = arrive(grp * nc + c, end_b);
                const int n_valid = min(kPcKeys, n_keys - c * kPcKeys), j0 = k_begin + c * kPcKeys + warp * 16;
                if (warp * 16 >= n_valid) continue;
                uint32_t mark[2] = {0u, 0u};                  // keys lane / 4 and lane / 4 + 8
                {
                    const float A = split_amax(pc_tile_amax<D>(buf + warp * 16 * kRow, lane));
                    const uint32_t tile = smem_addr(buf) + warp * 16 * kRow;
                    uint32_t a[D / 16][4];
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) ldmatrix_x4(a[kk], tile + (klane ^ (kk << 5)));
                    for (int o = 0; o < cnt; ++o) {
                        float acc[4] = {0.f, 0.f, 0.f, 0.f}, acc2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk) {
                            const uint2 q = fr[(o * (D / 16) + kk) * 32 + lane];
                            mma16816(kk & 1 ? acc2 : acc, a[kk], q.x, q.y);
                        }
                        const int r0 = o * 8 + 2 * (lane & 3);
                        uint32_t open = 0u;
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int row = oct0 * 8 + r0 + (x & 1), qpos = R.pos(row), j = j0 + (lane >> 2) + (x >> 1) * 8;
                            const float margin = (acc[x] + acc2[x]) - misc->thr_f[r0 + (x & 1)];
                            const float err = misc->err_f[r0 + (x & 1)] * A + misc->slack[r0 + (x & 1)];
                            const bool on = j < k_end && j < qpos;
                            if (on && margin >= err) mark[x >> 1] = pc_join(w, mark[x >> 1], pc_mark(w, R.rho(row), qpos));
                            else if (on && margin > -err) open |= 1u << x;
                        }
                        if (__any_sync(0xffffffffu, open != 0u))
                            pc_open_verdicts<T, D>(p, R, Qu, Ku, j0, oct0 * 8 + o * 8, open, thr_sm, qe_sm, eps_unit, flags, misc, mark);
                    }
                }
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    mark[y] = pc_join(w, mark[y], __shfl_xor_sync(0xffffffffu, mark[y], 1));
                    mark[y] = pc_join(w, mark[y], __shfl_xor_sync(0xffffffffu, mark[y], 2));
                    const int j = j0 + (lane >> 2) + y * 8;
                    if ((lane & 3) == 0 && j < k_end) words_g[j] = grp ? pc_join(w, words_g[j], mark[y]) : mark[y];   // the same lane's
                }
            }
        }
    } else {
        for (int c = 0; c < nc; ++c) {
            if (tid < kPcKeys) words_sm[tid] = 0u;
            const unsigned char* buf = arrive(c, end_b);
            const int n_valid = min(kPcKeys, n_keys - c * kPcKeys);
            if (works)
                for (int ru = my_ru; ru < n_ru; ru += ru_slots) {
                    if (!keep_rows) stage_rows(ru);
                    for (int sub = my_kg; sub < kSubs && sub * 32 < n_valid; sub += key_groups) {
                        double acc[4];
                        const int kr = sub * 32 + lane, j = k_begin + c * kPcKeys + kr;
                        dot4(buf, kr, acc);
                        uint32_t mark = 0u;
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int row = ru * 4 + x, qpos = R.pos(row);
                            if (j >= k_end || j >= qpos) continue;
                            const double th = thr_sm[row], margin = acc[x] * inv_root_d - th, e = th > -INFINITY ? 1e-13 * (1.0 + fabs(th)) : 0.0;   // (alpha = 0: all important)
                            if (margin > e) mark = pc_join(w, mark, pc_mark(w, R.rho(row), qpos));
                            else if (margin >= -e) pc_leave_open(flags, misc, row, j);               // a tie (a query at position 1)
                        }
                        if (mark) {
                            if (w <= 32) atomicOr(words_sm + kr, mark);
                            else atomicMax(words_sm + kr, mark);
                        }
                    }
                }
            __syncthreads();
            if (tid < n_valid) words_g[k_begin + c * kPcKeys + tid] = words_sm[tid];
        }
    }
    __syncthreads();
    if constexpr (kTc) {
        if (warp == 0) tc_free(block.tmem);
        if (block.late) report_status(p.status, CORM_ERR_TIMEOUT);
    }

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

// Whether phases A and B of a bf16 pass run on tcgen05. The time there follows the groups of 128 rows, on mma.sync the rows, so what
// counts is how full the groups are; short prompts and few units (whose clusters of eight are resident at once) gain in any
// case. Time on mma.sync over that on tcgen05, equal prompts of 1000 to 8000 keys, 24 to 512 units, 128 / 64 channels:
//   rows   96 0.87-1.32 / 0.85-1.26   112 0.97-1.48 / 0.90-1.60   128 1.02-1.49 / 1.09-1.51   129 0.81-1.14 / 0.76-1.04
//         144 0.80-1.10 / 0.75-1.05   160 0.88-1.20 / 0.82-1.15   192 0.99-1.37 / 0.90-1.32   224 1.11-1.66 / 1.06-1.52
//         256 1.30-1.78 / 1.01-1.61
// 256 to 500 keys: 0.96 and more, 96 units x 256 keys 1.7-3.4; 1 to 12 units of any length: 0.86-2.1, 1.3 in the mean. 1024 units
// x 3000 keys, 100 rows, 3760 -> 3070 us.
inline bool tc_takes(int n_units, int rows, int max_p, int sm_count) {
    if (rows < kTcMinRows || rows > kTcMaxRows || max_p < 256) return false;
    const int groups = (rows + kTcRows - 1) / kTcRows;
    const double fill = (double)rows / (groups * kTcRows);
    if (max_p <= 512 || n_units * 148 <= 15 * sm_count || fill >= 0.9) return true;
    return groups > 1 ? fill >= 0.72 : (double)n_units * max_p * rows >= 2e8;
}

// Blocks per unit on tcgen05 (one per SM; 33 clusters of four and 15 of eight are resident at once): those that let the pass
// end first, a block costing 160 keys beside its own. Equal prompts take whole waves; of ragged ones the last wave is half full
// in the mean. us per pass with 1 / 2 / 4 / 8 blocks, 128 channels unless said otherwise:
//   256 rows, 3000 keys, 40 units 774 / 443 / 470 / 393, 64 units 784 / 453 / 489 / 599, 72 units 785 / 456 / 656 / 628; 2048..4096
//   keys, 75 units 942 / 741 / 649 / 691, 96 units 958 / 800 / 705 / 898, 124 units 1014 / 895 / 905 / 1084, 128 units 994 / 908
//   / 932 / 1174; 1500..3000 keys, 200 units 1192 / 978 / 1097 / 1437, 320 units 1581 / 1407 / 1653 / 2235; 128 units x 256 keys 115
//   / 169 / 281, 80 x 500 172 / 174 / 179 / 277, 120 x 1000 329 / 340 / 388 / 519; 800..1600 keys, 496 units 1299 / 1255 / 1656
//   100 rows, 512 x 3000 1767 / 1706 / 2212 / 2566; 512 rows, 80 x 4096 1981 / 1948 / 1554 / 1678; 64 channels, 80 x 3000 583 /
//   570 / 475 / 515. Off by the most: 16 units x 8192 keys, 128 rows, 1134 / 603 / 344 / 330 (four).
inline int tc_blocks_per_unit(int n_units, int mean_p, int max_p, int n_words, int sm_count) {
    const double sms = sm_count > 0 ? sm_count : 148, resident[4] = {sms, sms / 2, sms * 33 / 148, sms * 15 / 148};
    const double ragged = std::min(1.0, 4.0 * (max_p - mean_p) / std::max(1, max_p));
    int best = 1;
    double least = 0.0;
    for (int i = 0, cs = 1; cs <= kPcMaxCluster && cs <= n_words; ++i, cs *= 2) {
        const double waves = n_units / resident[i], longest = 160.0 + (double)max_p / cs, last = std::ceil(waves) - waves;
        const double cost = waves <= 1.0 ? longest : waves * (160.0 + (double)mean_p / cs) + (last + ragged * (0.5 - last)) * longest;
        if (cs == 1 || cost < least) { best = cs; least = cost; }
    }
    return best;
}

// Host side. Returns CORM_ERR_UNSUPPORTED when the launch does not fit. mean_p: tokens of a prompt in the mean.
template <typename T, int D, bool kTc = false>
inline corm_status_t launch_prompt_cluster(const PromptParams& p, int G, int mean_p, int max_p, int sm_count, cudaStream_t st) {
    if constexpr (!kTc && Elem<T>::kBytes == 2)
        if (tc_takes(p.U, p.w * G, max_p, sm_count)) return launch_prompt_cluster<T, D, true>(p, G, mean_p, max_p, sm_count, st);
    PromptClusterParams pp{};
    pp.p = p;
    while ((1 << pp.log2g) < G) ++pp.log2g;
    pp.rows8 = (p.w * G + 7) / 8 * 8;
    const int n_words = std::max(1, (max_p + 31) / 32);
    // As many blocks per unit as make the launch at least five waves of resident blocks: fewer leave the machine
    // to the longest units, more pay each block's fixed chain of round trips more often (on tcgen05: tc_blocks_per_unit). us per
    // pass with 1 / 2 / 4 / 8, on the first version of the kernel (the shapes take 840, 598 and 60 us now, with 2, 8 and 8):
    // 1024 units x 3250 keys 969-1353 (with the slab's stride) / 956-1033 / 1073 / 1365, 128 units x 8192 keys (G 4) 2152 / 1281 / 811 / 752, 32 units x
    // 4096 keys 350 / 192 / 120 / 93.
    int cs = 1;
    if constexpr (kTc) cs = tc_blocks_per_unit(p.U, mean_p, max_p, n_words, sm_count);
    else while (cs < kPcMaxCluster && cs * 2 <= n_words && (long long)p.U * cs < 1500ll * sm_count / 148) cs *= 2;
    PcSmem lay;
    if constexpr (kTc) lay = tc_smem_layout<D>(pp.rows8); else lay = pc_smem_layout<T, D>(pp.rows8);
    if (lay.total > 227 * 1024) return CORM_ERR_UNSUPPORTED;
    auto kern = prompt_cluster_kernel<T, D, kTc>;
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), (size_t)lay.total);
    if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)p.U, (unsigned)cs);
        cfg.blockDim = dim3(kTc ? kTcThreads : kPcThreads);
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
