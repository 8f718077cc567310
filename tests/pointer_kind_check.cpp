// Which memory kernels read in place (see test_pointer_kind_host.py).
#include <cstdio>
#include <initializer_list>

#include "pointer_kind.h"

using namespace snp;

int main() {
    int bad = 0;
    for (int dev : {0, 1, 7})
        for (int owner : {0, 1, 7}) {
            for (cudaMemoryType t : {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged}) {
                cudaPointerAttributes a{};
                a.type = t;
                a.device = owner;
                const bool gpu = t == cudaMemoryTypeDevice || t == cudaMemoryTypeManaged;
                bad += is_device_memory(a) != gpu;
                bad += readable_in_place(a, dev) != (gpu && owner == dev);
            }
        }
    std::printf("bad=%d\n", bad);
    return bad;
}
