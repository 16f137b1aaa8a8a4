// What a test sets and reads of the host-only CUDA runtime (fake_cudart.cpp).
#pragma once

#include <string>
#include <vector>

struct Fake {
    int device = 0;
    bool refuse_attributes = false;
    std::vector<std::string> launched;  // kernels, mangled
    std::vector<void*> streams;         // their streams
};
extern Fake fake;
