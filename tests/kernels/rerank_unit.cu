// The rerank kernel by itself, for tests: records, candidates and queries of the caller's, and the limit of
// a wait as a parameter.
#include "../../paper_2312_16335_gb300/csrc/rerank.cu"

namespace lv {
int fail(int code, const std::string &) { return code; }
int cuda_fail(cudaError_t, const char *) { return LV_ERR_CUDA; }
}  // namespace lv

extern "C" int rerank_unit(const uint8_t *sec, int64_t stride, int chunks, int bits, int metric, const float *Q,
                           int64_t m, int D, const float *smean, const int32_t *cand, const int *cand_n, int ldc, int k,
                           int32_t *ids, float *scores, int ldo, int *status, int tries, void *stream) {
    using namespace lv;
    BeamParams bp;
    memset(&bp, 0, sizeof(bp));
    bp.sec = sec;
    bp.sec_stride = stride;
    bp.sec_chunks = chunks;
    bp.sec_bits = bits;
    bp.metric = metric;
    bp.Q = Q;
    bp.D = D;
    bp.smean = smean;
    bp.uni = make_int4(k, ldc, ldc, 0);
    bp.m = m;
    bp.cand = const_cast<int32_t *>(cand);
    bp.cand_n = const_cast<int *>(cand_n);
    bp.ldc = ldc;
    bp.ids = ids;
    bp.scores = scores;
    bp.ldo = ldo;
    bp.status = status;
    return launch_rerank(bp, (cudaStream_t)stream, tries);
}
