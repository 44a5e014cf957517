// The shape and shared-memory limit of the neighbour build (build_group_shape) on a machine made up
// by fake_cudart.cpp.  usage: build_shape_check <mode> <cap> <mean neighbours>
// <neighbours in the densest liquid>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <utility>

#include "gbmd_internal.cuh"

extern int fake_device, fake_refuse;
extern std::map<std::pair<int, const void*>, int> fake_limit;

int main(int, char** argv)
{
    using namespace gbmd;
    Scal S{};
    Launch L{};
    S.mode = std::atoi(argv[1]);
    S.cap = std::atoi(argv[2]);
    L.nsm = 152;
    const double mean = std::atof(argv[3]), dense = std::atof(argv[4]);
    // the limit must reach what a launch asks for on every device a system is made on
    int bad = 0;
    for (int round = 0; round < 2; ++round)
        for (fake_device = 0; fake_device < 3; ++fake_device)
            for (S.half_list = 0; S.half_list < (S.mode == MD_FP64 ? 1 : 2); ++S.half_list) {
                fake_limit.clear();
                if (build_group_shape(S, L, mean, dense, 232448) != cudaSuccess) ++bad;
                if (fake_limit.size() != 1 || fake_limit.begin()->first.first != fake_device ||
                    fake_limit.begin()->second < L.bg_smem)
                    ++bad;
            }
    S.half_list = 0;
    fake_refuse = 1;
    if (build_group_shape(S, L, mean, dense, 232448) == cudaSuccess) ++bad;     // a refusal reaches the caller
    std::printf("rows %d warps %d smem %d bad %d\n", L.bg_rows, L.bg_block / 32, L.bg_smem, bad);
    return 0;
}
