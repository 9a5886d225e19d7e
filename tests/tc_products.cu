// The products of phase A and B of the prompt pass on tcgen05, as corm_prompt_tc.cuh forms them, on operands of the caller's.
#include "../paper_2404_15949_b200/csrc/corm_prompt_tc.cuh"

using namespace corm;

// rows: q1, q2, q3 and the raw values, [4][128][D] bf16; keys: k1, k2, r2 and the raw values, [4][64][D]; out: [5][128][64], the
// four accumulators of phase A and the one of phase B
template <int D>
__global__ void __launch_bounds__(256) products(const uint4* rows, const uint4* keys, float* out, int* status) {
    using S = TcShape<D>;
    constexpr int kC = D / 8, kKeysAt = 4 * S::kRowPiece, kMiscAt = kKeysAt + 4 * S::kKeyPiece;
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(smem + kMiscAt);
    uint32_t* tmem = reinterpret_cast<uint32_t*>(smem + kMiscAt + 16);
    auto place = [](int r, int c, int block) { return (c >> 3) * block + r * 128 + (((c & 7) ^ (r & 7)) << 4); };
    for (int x = tid; x < 4 * kTcRows * kC; x += 256) {
        const int piece = x / (kTcRows * kC), r = x / kC % kTcRows, c = x % kC;
        *reinterpret_cast<uint4*>(smem + piece * S::kRowPiece + place(r, c, S::kRowBlock)) = rows[x];
    }
    for (int x = tid; x < 4 * kTcKeys * kC; x += 256) {
        const int piece = x / (kTcKeys * kC), r = x / kC % kTcKeys, c = x % kC;
        *reinterpret_cast<uint4*>(smem + kKeysAt + piece * S::kKeyPiece + place(r, c, S::kKeyBlock)) = keys[x];
    }
    if (tid == 0) { mbar_init(smem_addr(bar), 1); fence_mbar_init(); }
    if (warp == 0) tc_alloc(smem_addr(tmem));
    fence_async_smem();
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    const uint32_t d = *tmem;
    if (tid == 0) {
        const uint32_t q1 = smem_addr(smem), q2 = q1 + S::kRowPiece, q3 = q2 + S::kRowPiece, q = q3 + S::kRowPiece;
        const uint32_t k1 = smem_addr(smem + kKeysAt), k2 = k1 + S::kKeyPiece, r2 = k2 + S::kKeyPiece, k = r2 + S::kKeyPiece;
        tc_product<D>(d, q1, k1, false);
        tc_product<D>(d + 64, q2, k1, false);
        tc_product<D>(d + 64, q1, k2, true);
        tc_product<D>(d + 128, q2, k2, false);
        tc_product<D>(d + 192, q3, k1, false);
        tc_product<D>(d + 192, q2, r2, true);
        tc_product<D>(d + 192, q1, r2, true);
        tc_product<D>(d + 256, q, k, false);
        tc_commit(smem_addr(bar));
    }
    if (!mbar_wait(smem_addr(bar), 0)) *status = 1;
    tc_after_sync();
    if (warp < 4)
        for (int a = 0; a < 5; ++a)
            for (int g = 0; g < 8; ++g) {
                uint32_t v[8];
                tc_load8(v, d + ((uint32_t)(warp * 32) << 16) + a * 64 + g * 8);
                tc_wait_loads();
                tc_loaded(v);
                for (int k = 0; k < 8; ++k) out[(a * kTcRows + warp * 32 + lane) * kTcKeys + g * 8 + k] = __uint_as_float(v[k]);
            }
    tc_before_sync();
    __syncthreads();
    if (warp == 0) tc_free(d);
}

template <int D> static int run(const void* rows, const void* keys, void* out, void* status) {
    using S = TcShape<D>;
    constexpr int kBytes = 4 * S::kRowPiece + 4 * S::kKeyPiece + 64, kAsk = kBytes > kTcMinSmem ? kBytes : kTcMinSmem;
    static_assert(kAsk <= 227 * 1024, "operands fit");
    if (cudaFuncSetAttribute(products<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAsk) != cudaSuccess) return 1;
    products<D><<<1, 256, kAsk>>>(static_cast<const uint4*>(rows), static_cast<const uint4*>(keys), static_cast<float*>(out), static_cast<int*>(status));
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}
extern "C" int tc_products(int head_dim, const void* rows, const void* keys, void* out, void* status) {
    return head_dim == 128 ? run<128>(rows, keys, out, status) : run<64>(rows, keys, out, status);
}
