// What both forms of the prompt-end pass share (corm_prompt.cuh, corm_prompt_tc.cuh): block and chunk sizes, the layout of
// shared memory, the rows of a unit, marks and open verdicts.
#pragma once

#include "corm_mma.cuh"

namespace corm {

constexpr int kPcThreads = 256;
constexpr int kPcWarps = kPcThreads / 32;
constexpr int kPcKeys = 128;                    // keys per ring buffer
// ring buffers: three, two where rows are long or the row pieces of a group take the room
template <typename T, int D> __host__ __device__ constexpr int pc_bufs(int rows8) {
    return D * Elem<T>::kBytes > 256 || (Elem<T>::kBytes == 2 && D == 128 && rows8 > 16) ? 2 : 3;
}
constexpr int kPcGroup = 4;                     // octets of rows (bf16) whose pieces lie on chip at a time in phase A
constexpr int kPcGroupB = 8;                    // ... whose raw values do in phase B
constexpr int kPcMaxCluster = 8;
constexpr double kPcLogitLimit = 650.0;         // exp of anything below stays finite in fp64, also summed over 2^19 keys

struct PcSmem { int ring, zs, thr, n1, qe, flags, words, list, stage, frag, misc, tc, total; };
constexpr int kPcOpenCap = 64;
struct PcMisc {
    double red[kPcWarps][2];
    double mz[2];
    double zw[kPcWarps][kPcGroup * 8];          // phase A: the warps' sums of a group's rows
    int count, bad, warp_sum[kPcWarps], fail;
    int n_open;                                 // verdicts that phase B left open: (row, key)
    int2 open[kPcOpenCap];
    uint32_t amax;                              // largest magnitude (bf16 bits) of the block's keys
    float thr_f[kPcGroupB * 8], err_f[kPcGroupB * 8], slack[kPcGroupB * 8];      // phase B: a group's rows
};

__device__ __forceinline__ void cp_async16_zfill(uint32_t dst_smem, const void* src_gmem, bool on) {
    const int n = on ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst_smem), "l"(src_gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

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

__device__ __forceinline__ void pc_leave_open(uint32_t* flags, PcMisc* misc, int row, int j) {
    atomicOr(flags + (row >> 5), 1u << (row & 31));
    const int at = atomicAdd(&misc->n_open, 1);
    if (at < kPcOpenCap) misc->open[at] = make_int2(row, j);
}

}  // namespace corm
