// fan.hpp -- side streams on which the cluster-mode waves of a batched or served step
// run beside its cooperative ones.
//
// Every wave of a step works on images of its own, so the order between them is
// free.  A cluster is scheduled whole and waits for no other launch, so cluster
// waves may overlap each other and a cooperative wave; cooperative waves stay in
// one chain, since two of them may not be resident together.  24 uneven images
// launch up to 13 cluster waves a step, each a few blocks for 30-70 us.
#pragma once

#include <cuda_runtime.h>

namespace eecmg {

class Fan {
public:
    static constexpr int SIDES = 8;
    // Makes up to n side streams and their events, all that this fan will ever have: a
    // capture and a serving thread make none.  What cannot be made is done without.
    void create(int n);
    void destroy();
    // Queues a cluster launch on the next side stream (on s where there is none);
    // begin() forks the side streams off s at their first use, end() joins those used
    // back into s.
    void begin(cudaStream_t s);
    cudaError_t next(cudaStream_t* out);
    cudaError_t end();

private:
    cudaStream_t side_[SIDES] = {};
    cudaEvent_t fork_ = nullptr, join_[SIDES] = {};
    int made_ = 0;  // side streams
    cudaStream_t main_ = nullptr;
    int n_ = 0;     // cluster launches so far
    int used_ = 0;  // side streams forked off main_
};

}  // namespace eecmg
