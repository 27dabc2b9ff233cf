"""Which of the caller's vectors sim_apply_shifted's kernel uses where they lie:
its own device's memory and managed memory, aligned; another GPU's memory, host
memory and unregistered pointers take the copies."""
import native_program


def test_in_place_only_for_memory_the_kernel_can_reach(tmp_path):
    out = native_program.run(tmp_path, r'''
#include <cstdio>
#include "in_place.h"
int main() {
    for (int dev = 0; dev < 2; ++dev)
        for (int type : {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged})
            for (int device = 0; device < 2; ++device)
                for (long at : {4096l, 4104l}) {
                    cudaPointerAttributes a{};
                    a.type = (cudaMemoryType)type;
                    a.device = device;
                    printf("%d %d %d %ld %d\n", dev, type, device, at, (int)sim::usable_in_place(a, dev, (void*)at));
                }
}
''')
    rows = [tuple(map(int, r.split())) for r in out.splitlines()]
    assert len(rows) == 32
    for dev, kind, device, at, used in rows:
        # 2: device memory, 3: managed
        assert used == int(at % 16 == 0 and ((kind == 2 and device == dev) or kind == 3)), (dev, kind, device, at)
