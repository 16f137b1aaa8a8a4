"""Host code against a CUDA runtime that is not there: the library's own objects linked with
fake_cudart.cpp, which keeps a kernel's attributes per device, refuses calls on demand and
records the launches.  No GPU is used."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def build(tmp_path_factory):
    from paper_2311_03010_gb300 import build_lib

    build_lib.build()
    d = tmp_path_factory.mktemp("host")
    cuda = os.path.join(os.path.dirname(os.path.dirname(build_lib._nvcc())), "include")
    if not os.path.isdir(cuda):
        cuda = "/usr/local/cuda/include"
    fake = str(d / "fake.o")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", cuda, "-c", os.path.join(HERE, "fake_cudart.cpp"), "-o", fake], check=True)

    def run(name, source, objects):
        src, obj, exe = (str(d / (name + e)) for e in (".cu", ".o", ""))
        with open(src, "w") as f:
            f.write('#include <cstdio>\n#include <cstdlib>\n#include "fake_cudart.h"\n'
                    '#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\\n", __LINE__, #x); std::exit(1); } } while (0)\n' + source)
        subprocess.run([build_lib._nvcc()] + build_lib.ARCH + ["-std=c++17", "--expt-relaxed-constexpr", "-I", HERE, "-I", build_lib.CSRC,
                                                              "-c", src, "-o", obj], check=True)
        subprocess.run(["g++", obj, fake] + [os.path.join(build_lib.BUILD, o + ".o") for o in objects] + ["-o", exe], check=True)
        r = subprocess.run([exe], capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr

    return run


def test_large_tiles_on_a_second_device_and_after_a_refusal(build):
    build("wide", r'''
#include "launch.hpp"
using namespace eecmg;
static std::string apply(int device) {
    fake.device = device;
    fake.launched.clear();
    float x = 0, y = 0;
    Taps t{};
    ConvArgs a;
    a.x = &x;
    a.y = &y;
    a.taps = &t;
    a.h = 900;
    a.w = 2280;
    for (int r = 0; r <= EECMG_MAX_RADIUS; ++r) CHECK(launch_conv(a, r, 1, 0, nullptr) == cudaSuccess);
    CHECK(fake.launched.size() == EECMG_MAX_RADIUS + 1);
    for (auto& n : fake.launched) CHECK((n.find("k_conv_wide") != n.npos) == (fake.launched[0].find("k_conv_wide") != n.npos));
    return fake.launched[0];
}
int main() {
    CHECK(apply(0).find("k_conv_wide") != std::string::npos);
    CHECK(apply(1).find("k_conv_wide") != std::string::npos);
    fake.refuse_attributes = true;  // the small tiles need none
    CHECK(apply(2).find("k_conv_wide") == std::string::npos);
    CHECK(cudaGetLastError() == cudaSuccess);
    fake.refuse_attributes = false;
    CHECK(apply(2).find("k_conv_wide") != std::string::npos);
    return 0;
}
''', ["conv.cu"])


def test_clusters_on_a_second_device_and_after_a_refusal(build):
    build("clusters", r'''
#include "level_solve.hpp"
namespace eecmg {
cudaError_t launch_level_cgls_f32_lo(const LevelLaunch& L, int rt, int sep, int prec, int op, int blocks, cudaStream_t s, int* out);
}
using namespace eecmg;
static cudaError_t solve(int device, int op) {  // 16 blocks to a cluster, two tiles each where resident
    fake.device = device;
    fake.launched.clear();
    LevelLaunch L;
    L.cluster = 16;
    L.resident = op == LS_RESIDENT ? 2 : 0;
    const cudaError_t e = launch_level_cgls_f32_lo(L, 3, 1, 0, op, 16, nullptr, nullptr);
    cudaGetLastError();
    CHECK((fake.launched.size() == 1) == (e == cudaSuccess));
    return e;
}
int main() {
    for (int op : {LS_RESIDENT, LS_CLUSTER}) {
        for (int device : {0, 1, 0}) CHECK(solve(device, op) == cudaSuccess);
        fake.refuse_attributes = true;
        CHECK(solve(2, op) != cudaSuccess);
        fake.refuse_attributes = false;  // a refusal is not remembered
        CHECK(solve(2, op) == cudaSuccess);
    }
    return 0;
}
''', ["ls_cgls_f32_lo.cu"])


def test_side_streams_are_made_once_and_done_without(build):
    build("fan", r'''
#include <set>
#include "fan.hpp"
using namespace eecmg;
static std::vector<cudaStream_t> waves(Fan& f, cudaStream_t s, int n) {
    std::vector<cudaStream_t> got(n);
    fake.waits.clear();
    f.begin(s);
    for (auto& t : got) CHECK(f.next(&t) == cudaSuccess);
    CHECK(f.end() == cudaSuccess);
    return got;
}
int main() {
    cudaStream_t s = (cudaStream_t)0x1000;
    for (int want : {0, 1, 3, Fan::SIDES}) {
        for (int limit : {0, 1, 2, 100}) {  // streams that can be made
            Fan f;
            fake.streams_left = limit;
            f.create(want);
            CHECK(cudaGetLastError() == cudaSuccess);
            const int made = fake.made;
            const int sides = want < limit ? want : limit;
            for (int n : {0, 1, 2, 5, 20}) {
                const auto got = waves(f, s, n);
                const std::set<cudaStream_t> used(got.begin(), got.end());
                CHECK((int)used.size() == (sides == 0 ? (n > 0) : n < sides ? n : sides));
                if (sides == 0) CHECK(n == 0 || *used.begin() == s);
                // every side stream used waits for the main one, and the main one for each
                CHECK(fake.waits.size() == (sides == 0 ? 0 : 2 * used.size()));
                for (size_t i = 0; i < fake.waits.size(); ++i) CHECK((fake.waits[i] == s) == (i >= used.size()));
            }
            CHECK(fake.made == made);  // nothing made after create()
            f.destroy();
            CHECK(fake.made == 0);
        }
    }
    return 0;
}
''', ["fan.cpp"])
