// Host check of what the server and svm_train_batch tell of a job by the
// record that the batch kernel left (batch_status.cuh).
#include <cstdint>
#include <cstdio>

#include "batch_status.cuh"

using namespace svmgb;

struct Record {   // BatchResultDev's fields
    double b, b_up, b_low, objective;
    int64_t iters;
    int32_t status, n_sv;
};

int main()
{
    int bad = 0;
    auto expect = [&](int status, int rc, bool filled) {
        const Record R = {1.5, 2.5, 3.5, 4.5, 7, status, 9};
        svm_result r = {-1, -1, -1, -1, -1, -1, -1};
        const int got = job_result(R, r);
        const bool full = r.b == 1.5 && r.b_up == 2.5 && r.b_low == 3.5 && r.objective == 4.5 && r.iters == 7 && r.n_sv == 9;
        const bool none = r.b == 0 && r.b_up == 0 && r.b_low == 0 && r.objective == 0 && r.iters == 0 && r.n_sv == 0;
        if (got != rc || r.status != rc || (filled ? !full : !none)) {
            std::printf("status %d: got %d, want %d\n", status, got, rc);
            ++bad;
        }
    };
    expect(0, SVM_OK, true);
    expect(1, SVM_NOT_CONVERGED, true);
    expect(2, SVM_ERR_TIMEOUT, false);
    expect(3, SVM_ERR_CUDA, false);
    expect(-1, SVM_ERR_CUDA, false);
    return bad != 0;
}
