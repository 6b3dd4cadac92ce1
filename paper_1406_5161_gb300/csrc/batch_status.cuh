// How a job of the batched solver ended (BatchResultDev::status), and what
// the callers of svm_train_batch and of the server are told. Host code only.
#pragma once

#include "svm_gb300.h"

namespace svmgb {

enum { JOB_CONVERGED = 0, JOB_ITER_LIMIT = 1, JOB_WAIT_GAVE_UP = 2 };

constexpr const char *kJobWaitMessage = "a wait in the batched SMO kernel exceeded its time limit";

// Only the two ends that leave a valid result are successes: whatever else a
// job reports, its multipliers are those of an unfinished solve.
inline int job_status(int code)
{
    switch (code) {
    case JOB_CONVERGED: return SVM_OK;
    case JOB_ITER_LIMIT: return SVM_NOT_CONVERGED;
    case JOB_WAIT_GAVE_UP: return SVM_ERR_TIMEOUT;
    default: return SVM_ERR_CUDA;
    }
}

// A served job's outcome from its result record: the fields that a caller
// reads only after SVM_OK or SVM_NOT_CONVERGED are filled for these alone.
// Record: b, b_up, b_low, objective, iters, status, n_sv (BatchResultDev).
template <class Record>
int job_result(const Record &R, svm_result &res)
{
    res = svm_result{};
    res.status = job_status(R.status);
    if (res.status < 0) return res.status;
    res.b = R.b;
    res.b_up = R.b_up;
    res.b_low = R.b_low;
    res.objective = R.objective;
    res.iters = R.iters;
    res.n_sv = R.n_sv;
    return res.status;
}

}  // namespace svmgb
