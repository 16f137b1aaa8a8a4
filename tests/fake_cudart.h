// What a test sets and reads of the host-only CUDA runtime (fake_cudart.cpp).
#pragma once

#include <string>
#include <vector>

struct Fake {
    int device = 0;
    bool refuse_attributes = false;
    std::vector<std::string> launched;  // kernels, mangled
    std::vector<void*> streams;         // their streams
    int streams_left = 1 << 30;         // streams that can still be made
    int made = 0;                       // streams and events alive
    std::vector<void*> waits;           // streams that wait for an event, in order
};
extern Fake fake;
