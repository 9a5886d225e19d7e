// Logits of bf16 keys on the tensor cores without giving up fp64 verdicts.
//
// A plain bf16 mma accumulates in fp32, which is not enough to decide Definition 3.1 near its threshold. Here both
// operands are cut into pieces on power-of-two grids so that the large partial products are whole numbers of one unit
// and their sums stay below 2^24 units: an fp32 accumulator then holds them exactly, whatever the order of additions.
//   key tile (16 keys, A = its largest magnitude, 2^e <= A < 2^(e+1), g = 2^(e-5)):
//     k = k1 + k2 + r2,  k1 a multiple of g with |k1| <= 64 g, k2 a multiple of g/128 with |k2| <= g/2, |r2| <= g/256
//   query row (Aq its largest magnitude, gq = 2^(eq-7)):
//     q = q1 + q2 + q3,  |q1| <= 256 gq, q2 a multiple of gq/512 with |q2| <= gq/2, |q3| <= gq/1024
//   k1.q1                      <= 128 * 64 * 256 units of g gq             = 2^21: exact
//   k1.q2 + k2.q1              <= 2^21 + 2^23 units of g gq / 512                  : exact, one accumulator
//   k2.q2 + r2.q1 + r2.q2 + k1.q3   rounded: fp32 sums of at most 68 terms per 16 channels
//   k2.q3 + r2.q3              left out: q3 is zero but for elements 2^10 smaller than the row's largest
// (checked on the GPU: 65536 chained sums each of up to 2^23.6 and within 2^24 - 1200..300 units, random and all of one
// sign, none off by a bit.)
// All pieces are exact bf16 numbers (rounding to a grid is an addition and a subtraction of 192 grid steps, two bf16
// instructions for two elements). The logit is the fp64 sum of the three accumulators; its error is bounded by
//   A (2^-17 (|q2|_1 / 64 + |q1|_1 / 8192 + |q3|_1) + |q3|_1 / 60)      (split_error below, 2^-17 = 64 roundings of 2^-23)
// which is about 3e-8 for unit normal rows of 128 channels after the 1/sqrt(d). Verdicts inside that bound are decided
// again in fp64 by the callers, so results never depend on it.
#pragma once

#include <cuda.h>

#include "corm_ptx.cuh"

namespace corm {

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst_smem, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst_smem), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x2_trans(uint32_t (&r)[2], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
// two floats -> one word of two bf16 (round to nearest even): `hi` in the upper half, `lo` in the lower
__device__ __forceinline__ uint32_t pack_bf16x2(float hi, float lo) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// the product without an addend
__device__ __forceinline__ void mma16816_zero(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ uint32_t add_bf16x2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("add.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t sub_bf16x2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// Elements of larger magnitude than 2^56 (or not finite) leave the range in which products of pieces are safe in fp32.
constexpr uint32_t kSplitMaxBits = (127u + 56u) << 7;          // bf16 bits of 2^56
constexpr uint32_t kSplitMinExp = 127u - 40u;                  // smaller tiles are cut on the grid of 2^-40

// The two grid constants (192 g and 192 g/128, each twice in a word) of a key tile whose largest magnitude has the
// bf16 bits `abits`.
struct SplitGrid { uint32_t m1, m2; };
__device__ __forceinline__ SplitGrid split_grid(uint32_t abits) {
    const uint32_t ex = max(abits >> 7, kSplitMinExp);
    const uint32_t c1 = ((ex + 2u) << 7) | 0x40u, c2 = ((ex - 5u) << 7) | 0x40u;
    return SplitGrid{c1 | (c1 << 16), c2 | (c2 << 16)};
}
// the tile's largest magnitude as the bound uses it
__device__ __forceinline__ float split_amax(uint32_t abits) { return __uint_as_float(max(abits, kSplitMinExp << 7) << 16); }

__device__ __forceinline__ void split_key(const uint32_t (&a)[4], SplitGrid g, uint32_t (&k1)[4], uint32_t (&k2)[4], uint32_t (&r2)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        k1[i] = sub_bf16x2(add_bf16x2(a[i], g.m1), g.m1);
        const uint32_t r = sub_bf16x2(a[i], k1[i]);
        k2[i] = sub_bf16x2(add_bf16x2(r, g.m2), g.m2);
        r2[i] = sub_bf16x2(r, k2[i]);
    }
}

// Pieces of one query element; c = 1.5 * 2^23 * gq of its row. Exact fp32 arithmetic.
__device__ __forceinline__ void split_query(float q, float c, float& q1, float& q2, float& q3) {
    const float c2 = c * (1.f / 512.f);
    q1 = __fsub_rn(__fadd_rn(q, c), c);
    const float r = __fsub_rn(q, q1);
    q2 = __fsub_rn(__fadd_rn(r, c2), c2);
    q3 = __fsub_rn(r, q2);
}
// c of split_query for a row whose largest magnitude is aq (finite, below 2^56)
__device__ __forceinline__ float split_query_const(float aq) {
    const int ex = max((int)((__float_as_uint(aq) >> 23) & 255u), 127 - 40);
    return __uint_as_float((uint32_t)(ex - 7 + 23) << 23) * 1.5f;
}
// error of a split logit (before the 1/sqrt(d)) per unit of the tile's largest magnitude; n1, n2, n3: 1-norms of the
// row and of its second and third pieces. The factor 1.2 covers the accumulators' own additions (4 of 64 and 8 of 128
// roundings), r2.q2 and the difference between the row's and its first piece's norm.
__device__ __forceinline__ float split_error(float n1, float n2, float n3) {
    return 7.62939453125e-6f * (n2 * (1.f / 64.f) + n1 * (1.f / 8192.f) + n3) * 1.2f + n3 * (1.f / 60.f);
}

// ---- exact logits ----
// A quarter of a row (lane's sub = lane & 3: the 16-byte chunks sub, sub + 4, ...) in registers, widened.
template <typename T, int D> struct QuadRow {
    static constexpr int kN = D / 4, kVec = 16 / Elem<T>::kBytes, kLoads = kN / kVec;
    double v[kN];
    __device__ __forceinline__ void load(const T* row, int sub) {
#pragma unroll
        for (int i = 0; i < kLoads; ++i) widen(__ldcg(reinterpret_cast<const uint4*>(row) + i * 4 + sub), i);
    }
    __device__ __forceinline__ void widen(const uint4& x, int i) {
        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if constexpr (kVec == 8) {
                v[i * 8 + 2 * e] = (double)__uint_as_float(w[e] << 16);
                v[i * 8 + 2 * e + 1] = (double)__uint_as_float(w[e] & 0xffff0000u);
            } else {
                v[i * 4 + e] = (double)__uint_as_float(w[e]);
            }
        }
    }
};
// N rows of the cache against one query, four lanes to a row: fp64, a fixed order (every caller gets the same bits for the
// same pair), before the 1/sqrt(d). Rows are read past the L1 (they move between launches that may overlap).
template <typename T, int D, int N>
__device__ __forceinline__ void quad_exact_dots(const QuadRow<T, D>& q, const T* const (&rows)[N], int sub, double (&s)[N]) {
    using Q = QuadRow<T, D>;
    uint4 x[N][Q::kLoads];
#pragma unroll
    for (int n = 0; n < N; ++n)
#pragma unroll
        for (int i = 0; i < Q::kLoads; ++i) x[n][i] = __ldcg(reinterpret_cast<const uint4*>(rows[n]) + i * 4 + sub);
#pragma unroll
    for (int n = 0; n < N; ++n) {
        double part = 0.0;
#pragma unroll
        for (int i = 0; i < Q::kLoads; ++i) {
            const uint32_t w[4] = {x[n][i].x, x[n][i].y, x[n][i].z, x[n][i].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if constexpr (Q::kVec == 8) {
                    part = fma(q.v[i * 8 + 2 * e], (double)__uint_as_float(w[e] << 16), part);
                    part = fma(q.v[i * 8 + 2 * e + 1], (double)__uint_as_float(w[e] & 0xffff0000u), part);
                } else {
                    part = fma(q.v[i * 4 + e], (double)__uint_as_float(w[e]), part);
                }
            }
        }
        part += __shfl_xor_sync(0xffffffffu, part, 1);
        part += __shfl_xor_sync(0xffffffffu, part, 2);
        s[n] = part;
    }
}
// Log-sum-exp of one query over the slots [begin + first, end) in steps of `step` by a whole warp, 16 slots at a time;
// row_of(j) gives a slot's row. All lanes return the same (m, Z).
template <typename T, int D, typename RowOf>
__device__ __forceinline__ void warp_exact_lse(const T* q, RowOf row_of, int begin, int end, int step, double& m, double& Z) {
    const int lane = threadIdx.x & 31, sub = lane & 3;
    QuadRow<T, D> qr;
    qr.load(q, sub);
    m = -INFINITY; Z = 0.0;
    for (int j0 = begin; j0 < end; j0 += step) {
        const int ja = j0 + (lane >> 2), jb = ja + 8;
        const T* const rows[2] = {row_of(min(ja, end - 1)), row_of(min(jb, end - 1))};
        double s[2];
        quad_exact_dots<T, D, 2>(qr, rows, sub, s);
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            if ((y ? jb : ja) >= end) continue;
            const double x = s[y] * inv_root_dim(D);
            if (x > m) { Z = Z * exp(m - x) + 1.0; m = x; }
            else Z += exp(x - m);
        }
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        const double mo = __shfl_xor_sync(0xffffffffu, m, o), Zo = __shfl_xor_sync(0xffffffffu, Z, o), mn = fmax(m, mo);
        Z = (m == mn ? Z : Z > 0.0 ? Z * exp(m - mn) : 0.0) + (mo == mn ? Zo : Zo > 0.0 ? Zo * exp(mo - mn) : 0.0);
        m = mn;
    }
}

// ---- clusters ----
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t cluster_size() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() { cluster_arrive(); cluster_wait(); }
// shared-memory address of the same variable in the cluster's block `rank`
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t ld_peer_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ld_peer_v4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ double ld_peer_f64(uint32_t addr) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
    return v;
}

// Pushes into the shared memory of a block of the cluster: value and byte count (on that block's barrier) arrive together.
__device__ __forceinline__ void push_u32(uint32_t addr, uint32_t v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void push_2u32(uint32_t addr, uint32_t x, uint32_t y, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(addr), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void push_v4(uint32_t addr, uint4 v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ void push_2f64(uint32_t addr, double x, double y, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];"
                 ::"r"(addr), "l"(__double_as_longlong(x)), "l"(__double_as_longlong(y)), "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_peer(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// mbar_wait for what other blocks of the cluster wrote
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity) {
    auto try_wait = [&]() -> bool {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        return ok != 0;
    };
    if (try_wait()) return true;
    const long long start = clock64();
    while (!try_wait())
        if (clock64() - start > kWaitLimitCycles) return false;
    return true;
}

}  // namespace corm
