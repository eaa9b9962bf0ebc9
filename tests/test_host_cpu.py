"""Rules and arithmetic of the library that the CPU can check. CPU only."""
from tests import host_cc


def test_only_memory_of_the_graphs_device_is_used_in_place(tmp_path):
    """Kernels take a caller's array in place only from their own device (or managed memory) and only
    aligned to its elements; a peer's memory, host memory and a byte offset are copied. An id array
    that shares bytes with a result is told apart from one that ends where the result begins."""
    out = host_cc.run(tmp_path, r"""
int main()
{
    auto at = [](uintptr_t a) { return reinterpret_cast<const void*>(a); };
    const cudaMemoryType D = cudaMemoryTypeDevice, M = cudaMemoryTypeManaged, H = cudaMemoryTypeHost,
                         U = cudaMemoryTypeUnregistered;
    printf("%d%d%d", rd::usable_in_place(D, 0, 0, at(4096), 8), rd::usable_in_place(D, 2, 2, at(4104), 8),
           rd::usable_in_place(M, 1, 0, at(4096), 8));
    printf("%d%d%d%d ", rd::usable_in_place(D, 1, 0, at(4096), 8), rd::usable_in_place(D, 0, 1, at(4096), 8),
           rd::usable_in_place(H, 0, 0, at(4096), 8), rd::usable_in_place(U, 0, 0, at(4096), 8));
    printf("%d%d%d ", rd::usable_in_place(D, 0, 0, at(4100), 8), rd::usable_in_place(D, 0, 0, at(4100), 4),
           rd::usable_in_place(M, 0, 0, at(4098), 4));
    printf("%d%d%d%d", rd::ranges_overlap(at(4096), 16, at(4108), 4), rd::ranges_overlap(at(4096), 16, at(4112), 4),
           rd::ranges_overlap(at(4112), 4, at(4096), 17), rd::ranges_overlap(at(4096), 16, nullptr, 4));
}
""", headers=("rd_internal.cuh",))
    assert out == "1110000 010 1010"
