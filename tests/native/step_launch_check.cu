// Launches every form of the CG step where no GPU can be reached (the caller hides the devices) and prints the errors that the
// launchers return: "<name> <cudaError_t>" per line. Nothing is read or written through the null pointers.
#include <cstdio>
#include <cstdlib>

#include "lgp_internal.cuh"

using namespace lgp;

int main() {
    const char *hidden = std::getenv("CUDA_VISIBLE_DEVICES");
    int devices = 0;
    if (!hidden || *hidden || (cudaGetDeviceCount(&devices) == cudaSuccess && devices > 0)) {
        std::puts("a GPU is visible");
        return 2;
    }
    (void)cudaGetLastError();
    CgBuffers b = {};
    b.G = 1;
    ProductTail none, few, many;
    few.S = 4;
    many.S = 40;
    few.part = many.part = reinterpret_cast<const float *>(16);
    CgSplit split = {};
    auto show = [](const char *name, cudaError_t e) {
        std::printf("%s %d\n", name, (int)e);
        (void)cudaGetLastError();
    };
    show("one-cta", launch_cg_after_matvec(1000, 1, b, none, nullptr, nullptr));
    show("cluster-8", launch_cg_after_matvec(30000, 1, b, few, nullptr, nullptr));
    show("three-vec4", launch_cg_after_matvec(300000, 4, b, none, nullptr, nullptr));
    show("three-vec4-parts", launch_cg_after_matvec(300000, 4, b, many, nullptr, nullptr));
    show("three-vec1", launch_cg_after_matvec(1000, 5, b, few, nullptr, nullptr));
    show("three-split", launch_cg_after_matvec(300000, 32, b, none, &split, nullptr));
    show("split", launch_p_split(split, nullptr, nullptr, 1000, 16, nullptr, nullptr));
    b.pc.k = 4;
    show("precond", launch_cg_after_matvec(1000, 4, b, none, nullptr, nullptr));
    show("precond-apply", launch_precond_apply(b.pc, nullptr, 1, nullptr, 1, nullptr, 1000, 1, nullptr, 1, nullptr, nullptr));
    show("tally", launch_cg_chunk_tally(nullptr, nullptr));
    return 0;
}
