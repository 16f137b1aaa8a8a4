// fan.cpp -- see fan.hpp.
#include "fan.hpp"

namespace eecmg {

void Fan::create(int n) {
    bool ok = n > 0 && cudaEventCreateWithFlags(&fork_, cudaEventDisableTiming) == cudaSuccess;
    while (ok && made_ < n && made_ < SIDES) {
        ok = cudaEventCreateWithFlags(&join_[made_], cudaEventDisableTiming) == cudaSuccess &&
             cudaStreamCreateWithFlags(&side_[made_], cudaStreamNonBlocking) == cudaSuccess;
        if (ok) ++made_;
    }
    if (n > 0 && !ok) cudaGetLastError();  // the waves share the streams there are
}

void Fan::destroy() {
    for (int i = 0; i < SIDES; ++i) {
        if (side_[i]) cudaStreamDestroy(side_[i]);
        if (join_[i]) cudaEventDestroy(join_[i]);
        side_[i] = nullptr;
        join_[i] = nullptr;
    }
    if (fork_) cudaEventDestroy(fork_);
    fork_ = nullptr;
    made_ = 0;
}

void Fan::begin(cudaStream_t s) {
    main_ = s;
    n_ = 0;
    used_ = 0;
}

cudaError_t Fan::next(cudaStream_t* out) {
    *out = main_;
    if (made_ == 0) return cudaSuccess;
    const int i = n_++ % made_;
    if (i == used_) {  // its first launch since begin()
        cudaError_t e = used_ == 0 ? cudaEventRecord(fork_, main_) : cudaSuccess;
        if (e == cudaSuccess) e = cudaStreamWaitEvent(side_[i], fork_, 0);
        if (e != cudaSuccess) return e;
        ++used_;
    }
    *out = side_[i];
    return cudaSuccess;
}

cudaError_t Fan::end() {
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < used_; ++i) {
        cudaError_t r = cudaEventRecord(join_[i], side_[i]);
        if (r == cudaSuccess) r = cudaStreamWaitEvent(main_, join_[i], 0);
        if (e == cudaSuccess) e = r;
    }
    used_ = 0;
    return e;
}

}  // namespace eecmg
