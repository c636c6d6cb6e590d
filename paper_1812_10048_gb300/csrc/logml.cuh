// Device state of a collapsed log-marginal-likelihood evaluation (fixed labels).
#pragma once

#include "common.cuh"

namespace dpmm {

struct LmlPlan {
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int num_sms = 0;
    int64_t N = 0;
    int32_t D = 0, K = 0;
    // inputs (device copies)
    int32_t* indptr = nullptr;
    int32_t* cols = nullptr;
    int32_t* counts = nullptr;
    int32_t* labels = nullptr;
    // statistics (scratch of the evaluation)
    uint32_t* n = nullptr;             // [K]
    uint32_t* S = nullptr;             // [K][D]
    unsigned long long* T = nullptr;   // [K]
    // scratch of k_lml_terms: per-block sums and the blocks that have finished
    // (zero between launches)
    double* part = nullptr;            // [lml_part_count(D)]
    int32_t* ticket = nullptr;
    // small outputs
    double* common = nullptr;          // sum_k [psi(B) - psi(B + T_k)]
    double* out = nullptr;             // [2]: logml, d/d log alpha
    float* grad = nullptr;             // [D] staging for host outputs
    float* beta_stage = nullptr;       // [D] staging for host inputs
};

cudaError_t lml_compute_stats(LmlPlan& p);
cudaError_t lml_stats_from_chain(LmlPlan& p, const uint32_t* nsub, const uint32_t* Ssub);
cudaError_t lml_stats_from_csr(LmlPlan& p, const Csr& csr, const int32_t* labels);
// The value (value_dev not null) and / or d/d log alpha with the constant that
// lml_backward needs (grad_alpha_dev not null).
// wrap_flag (may be null): kLmlWrapFlag is set in it when some T_k is 2^32 or
// more, so that a 32-bit gene total may have wrapped unseen.
constexpr uint32_t kLmlWrapFlag = 8u;
cudaError_t lml_terms(LmlPlan& p, double log_alpha, const float* log_beta, double* value_dev,
                      double* grad_alpha_dev, uint32_t* wrap_flag = nullptr);
cudaError_t lml_backward(LmlPlan& p, const float* log_beta, float* grad_dev);
size_t lml_part_count(int32_t D);   // doubles of LmlPlan::part

}  // namespace dpmm
