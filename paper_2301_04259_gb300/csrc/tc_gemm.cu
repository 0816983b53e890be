// tc_gemm.cu -- host side of the tcgen05 BF16 GEMM: tensor maps, tile choice, launch.
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "status_words.cuh"
#include "tc_gemm.cuh"

namespace soap {
namespace tc {

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// Row-major BF16 matrix [rows][cols] with row stride ld (elements), boxes of box_rows x 64.
soap_status operand_map(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    auto fn = encode_fn();
    if (!fn) { set_error("cuTensorMapEncodeTiled is not available from the driver"); return SOAP_ECUDA; }
    if ((reinterpret_cast<uintptr_t>(base) & 15) || (ld * 2) % 16 || ld < cols) {
        set_error("GEMM operand needs a 16-byte aligned base and a row stride that is a multiple of 8 elements");
        return SOAP_EINVAL;
    }
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
    cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { set_error("cuTensorMapEncodeTiled failed (%d)", (int)r); return SOAP_ECUDA; }
    return SOAP_OK;
}

soap_status encode_map(CUtensorMap* map, int rank, const void* base, const uint64_t* dims,
                       const uint64_t* strides, const uint32_t* box, CUtensorMapDataType dt) {
    auto fn = encode_fn();
    if (!fn) { set_error("cuTensorMapEncodeTiled is not available from the driver"); return SOAP_ECUDA; }
    if (rank < 1 || rank > 5 || (reinterpret_cast<uintptr_t>(base) & 15)) {
        set_error("tensor map: rank 1..5 and a 16-byte aligned base needed");
        return SOAP_EINVAL;
    }
    cuuint64_t d[5];
    cuuint64_t st[4];
    cuuint32_t bx[5], estr[5];
    for (int i = 0; i < rank; i++) {
        d[i] = (cuuint64_t)dims[i];
        bx[i] = (cuuint32_t)box[i];
        estr[i] = 1;
        if (i + 1 < rank) st[i] = (cuuint64_t)strides[i];
    }
    CUresult r = fn(map, dt, (cuuint32_t)rank, const_cast<void*>(base), d, st, bx, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { set_error("cuTensorMapEncodeTiled failed (%d)", (int)r); return SOAP_ECUDA; }
    return SOAP_OK;
}

template <int BN>
static soap_status launch(const CUtensorMap& ma, const CUtensorMap& mb, int M, int N, int K, const Epilogue& ep,
                          int sms, cudaStream_t st, unsigned int* flags) {
    static bool configured = false;     // per instantiation; attribute set is idempotent
    if (!configured) {
        SOAP_CUDA(cudaFuncSetAttribute(k_gemm_tn<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       Smem<BN>::kBytes));
        configured = true;
    }
    const int64_t tiles = (int64_t)((M + BM - 1) / BM) * ((N + BN - 1) / BN);
    k_gemm_tn<BN><<<(unsigned)std::min<int64_t>(tiles, sms), kThreads, Smem<BN>::kBytes, st>>>(ma, mb, M, N, K, ep, flags);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { set_error("GEMM launch failed: %s", cudaGetErrorString(e)); return SOAP_ECUDA; }
    return SOAP_OK;
}

soap_status gemm_tn(const __nv_bfloat16* A, int64_t lda, const __nv_bfloat16* B, int64_t ldb, int M, int N,
                    int K, const Epilogue& ep, cudaStream_t st, unsigned int* flags) {
    if (M <= 0 || N <= 0 || K <= 0) { set_error("GEMM sizes must be positive"); return SOAP_EINVAL; }
    int dev = 0, sms = 0;
    SOAP_CUDA(cudaGetDevice(&dev));
    SOAP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // 256 columns per tile read the fewest operand bytes per output; with fewer such tiles than SMs
    // narrower ones share the work out (7 x 16,834 x 384: 66 tiles of 256 columns, 132 of 128)
    const int64_t tiles_m = (M + BM - 1) / BM;
    const int BN = N <= 64 ? 64 : (N <= 128 || tiles_m * ((N + 255) / 256) < sms ? 128 : 256);
    CUtensorMap ma, mb;
    SOAP_TRY(operand_map(&ma, A, M, K, lda, BM));
    SOAP_TRY(operand_map(&mb, B, N, K, ldb, BN));
    if (BN == 64) return launch<64>(ma, mb, M, N, K, ep, sms, st, flags);
    if (BN == 128) return launch<128>(ma, mb, M, N, K, ep, sms, st, flags);
    return launch<256>(ma, mb, M, N, K, ep, sms, st, flags);
}

}  // namespace tc
}  // namespace soap

using namespace soap;

namespace soap {

// Status words of the entry points without a context, one per call in flight: so many calls at a time
// on all threads.
constexpr int kCallWords = 256;
static __device__ unsigned int g_call_words[kCallWords];
static StatusWords<kCallWords> g_call_status;

soap_status CallStatus::begin(unsigned int** word) {
    unsigned int* words = nullptr;
    SOAP_CUDA(cudaGetSymbolAddress((void**)&words, g_call_words));
    index_ = g_call_status.claim();
    word_ = words + index_;
    SOAP_CUDA(cudaMemsetAsync(word_, 0, sizeof(unsigned int), st_));
    *word = word_;
    return SOAP_OK;
}

soap_status CallStatus::finish(unsigned int* value) {
    SOAP_CUDA(cudaMemcpyAsync(value, word_, sizeof(unsigned int), cudaMemcpyDeviceToHost, st_));
    SOAP_CUDA(cudaStreamSynchronize(st_));
    done_ = true;
    return SOAP_OK;
}

CallStatus::~CallStatus() {
    if (index_ < 0) return;
    if (!done_) cudaStreamSynchronize(st_);          // its kernels may still write the word
    g_call_status.give_back(index_);
}

}  // namespace soap

extern "C" soap_status soap_gemm_bf16_tn(int32_t M, int32_t N, int32_t K, const void* A, int64_t lda,
                                         const void* B, int64_t ldb, const float* bias, int32_t activation,
                                         float* C, int64_t ldc, void* cuda_stream) {
    clear_error();
    if (!A || !B || !C) { set_error("NULL operand"); return SOAP_EINVAL; }
    if (activation != 0 && activation != 1) { set_error("activation must be 0 (none) or 1 (GELU)"); return SOAP_EINVAL; }
    if (ldc < N) { set_error("ldc < N"); return SOAP_EINVAL; }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    CallStatus status(st);
    unsigned int* flags = nullptr;
    SOAP_TRY(status.begin(&flags));
    tc::Epilogue ep{};
    ep.bias = bias;
    ep.gelu = activation;
    ep.c = C;
    ep.ldc = ldc;
    SOAP_TRY(tc::gemm_tn((const __nv_bfloat16*)A, lda, (const __nv_bfloat16*)B, ldb, M, N, K, ep, st, flags));
    unsigned int h = 0;
    SOAP_TRY(status.finish(&h));
    if (h) { set_error("GEMM kernel gave up waiting (status 0x%x)", h); return SOAP_ETIMEOUT; }
    return SOAP_OK;
}
