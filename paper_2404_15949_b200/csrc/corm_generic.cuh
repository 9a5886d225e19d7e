// Generic decode kernel: any supported dtype / head_dim / group size, written for clarity. One warp per key, lanes
// split the head dimension, fp64 logits. It serves corm_decode_step_static, whose scratch is a fixed array, and tuning
// value 0; every other step has a faster kernel.
#pragma once

#include "corm_common.cuh"

namespace corm {

constexpr int kGenericThreads = 128;

__host__ __device__ inline size_t generic_decode_smem(int D, int G, int C, bool paged) {
    const size_t warps = kGenericThreads / 32;
    size_t a = (size_t)G * D * 8 + warps * G * 16 + warps * G * D * 4;
    size_t b = (size_t)(paged ? 3 : 2) * ((C + 31) / 32 + 2) * 4;
    return a > b ? a : b;
}

// Decode step, one block per (split of a unit's live range, unit).
template <typename T, int D, int G>
__global__ void __launch_bounds__(kGenericThreads) decode_generic_kernel(const __grid_constant__ DecodeParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_last;
    constexpr int NT = kGenericThreads, NW = NT / 32, NPL = D / 32;
    const int u = blockIdx.y, split = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = u / p.Hkv;
    const int32_t* pt_u = p.page_table ? p.page_table + (size_t)u * p.pt_stride : nullptr;
    const int room = pt_u ? __ldcg(p.page_room + u) : 1;
    const int l_old = __ldcg(p.live_in + u), l = l_old + 1;
    if (l > p.C || !room) {   // the slab is full (paged: no page for the new row): report, leave the unit untouched
        if (split == 0 && tid == 0) { report_status(p.status, CORM_ERR_CAPACITY); p.live_out[u] = l_old; report_live(p, u, p.step + 1, l_old); }
        return;
    }
    const int n_act = (l + p.split_len - 1) / p.split_len;
    if (split >= n_act) return;
    const int t = __ldg(p.base_tokens + b) + p.step + 1;
    const int begin = split * p.split_len, end = min(l, begin + p.split_len);
    T* Kl = reinterpret_cast<T*>(p.K);                 // the layer's K / V storage: slabs or page pool
    T* Vl = reinterpret_cast<T*>(p.V);
    const size_t slab_row0 = (size_t)u * p.C;

    // append the current token (Algorithm 1's keys include it; its register starts at zero)
    if (l_old >= begin && l_old < end) {
        const T* kn = reinterpret_cast<const T*>(p.k_new) + (size_t)u * D;
        const T* vn = reinterpret_cast<const T*>(p.v_new) + (size_t)u * D;
        const size_t row = kv_row(pt_u, slab_row0, l_old, p.pool_pages, p.status);
        for (int c = tid; c < D; c += NT) { Kl[row * D + c] = kn[c]; Vl[row * D + c] = vn[c]; }
        if (Elem<T>::kBytes == 2 && warp == 0)
            note_key_magnitude(p.kmax + u, lane < D / 8 ? reinterpret_cast<const uint4*>(kn)[lane % (D / 8)] : make_uint4(0, 0, 0, 0));
        if (tid == 0) { p.word[(size_t)u * p.C + l_old] = 0u; p.pos[(size_t)u * p.C + l_old] = t; }
        __syncthreads();
    }

    double* qs = reinterpret_cast<double*>(smem);                      // [G][D]
    double* sm_mz = qs + G * D;                                        // [NW][G][2]
    float* sm_acc = reinterpret_cast<float*>(sm_mz + NW * G * 2);      // [NW][G][D]
    const T* qg = reinterpret_cast<const T*>(p.q) + (size_t)u * G * D;
    for (int i = tid; i < G * D; i += NT) qs[i] = (double)Elem<T>::load(qg + i);
    __syncthreads();

    const int c0 = lane * NPL;
    double qr[G][NPL];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int i = 0; i < NPL; ++i) qr[g][i] = qs[g * D + c0 + i];
    double m[G], Z[G];
    float acc[G][NPL];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        m[g] = -INFINITY; Z[g] = 0.0;
#pragma unroll
        for (int i = 0; i < NPL; ++i) acc[g][i] = 0.f;
    }
    const double root_d = sqrt((double)D);
    for (int j = begin + warp; j < end; j += NW) {
        float kf[NPL], vf[NPL];
        const size_t row = kv_row(pt_u, slab_row0, j, p.pool_pages, p.status);
        load_slice<T, NPL>(Kl + row * D + c0, kf);
        load_slice<T, NPL>(Vl + row * D + c0, vf);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            double part = 0.0;
#pragma unroll
            for (int i = 0; i < NPL; ++i) part += qr[g][i] * (double)kf[i];
            const double s = warp_sum(part) / root_d;                  // Eq. 2's exponent
            if (lane == 0) p.stash[((size_t)u * G + g) * p.C + j] = s;
            float pj;
            if (s > m[g]) {                                            // running-max softmax
                const double sc = exp(m[g] - s);
                Z[g] = Z[g] * sc + 1.0;
                const float scf = (float)sc;
#pragma unroll
                for (int i = 0; i < NPL; ++i) acc[g][i] *= scf;
                m[g] = s;
                pj = 1.f;
            } else {
                const double e = exp(s - m[g]);
                Z[g] += e;
                pj = (float)e;
            }
#pragma unroll
            for (int i = 0; i < NPL; ++i) acc[g][i] += pj * vf[i];     // Eq. 1
        }
    }
    // merge the warps of this block into one partial record per query head
#pragma unroll
    for (int g = 0; g < G; ++g) {
        if (lane == 0) { sm_mz[(warp * G + g) * 2] = m[g]; sm_mz[(warp * G + g) * 2 + 1] = Z[g]; }
#pragma unroll
        for (int i = 0; i < NPL; ++i) sm_acc[(warp * G + g) * D + c0 + i] = acc[g][i];
    }
    __syncthreads();
    const size_t pstride = partial_stride(D);
    for (int g = 0; g < G; ++g) {
        double M = -INFINITY;
        for (int w = 0; w < NW; ++w) M = fmax(M, sm_mz[(w * G + g) * 2]);
        double Zt = 0.0;
        unsigned char* rec = p.partials + (((size_t)u * p.max_splits + split) * G + g) * pstride;
        for (int c = tid; c < D; c += NT) {
            float a = 0.f;
            for (int w = 0; w < NW; ++w) a += sm_acc[(w * G + g) * D + c] * (float)exp(sm_mz[(w * G + g) * 2] - M);
            reinterpret_cast<float*>(rec + 16)[c] = a;
        }
        if (tid == 0) {
            for (int w = 0; w < NW; ++w) Zt += sm_mz[(w * G + g) * 2 + 1] * exp(sm_mz[(w * G + g) * 2] - M);
            reinterpret_cast<double*>(rec)[0] = M;
            reinterpret_cast<double*>(rec)[1] = Zt;
        }
    }
    // publish, then let the last-arriving split of this unit run the finalize phase
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        const unsigned prev = atomicAdd(p.ticket + u, 1u);
        s_last = (prev == (unsigned)(n_act - 1));
        if (s_last) p.ticket[u] = 0u;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    finalize_unit<T, D, G, NT>(p, u, b, l, n_act, t, smem);
}

}  // namespace corm
