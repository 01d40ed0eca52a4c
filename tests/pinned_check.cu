// Which host memory counts as one pinned range.  Without arguments: the ranges' arithmetic, on the host.  With one: what the
// driver says of allocations and registrations, two registrations with a hole between them among them.  Nothing but pointers
// is looked at; no kernel runs and no byte of the ranges is read.  Returns the number of answers that are wrong.
#include <stdio.h>
#include <sys/mman.h>

#include "impact_pinned.h"

using namespace impact;

static int bad = 0;
static void expect(bool got, bool want, const char* what) {
    if (got == want) return;
    ++bad;
    printf("%s: %d\n", what, (int)got);
}

int main(int argc, char**) {
    const auto at = [](unsigned long long a) { return reinterpret_cast<const void*>((uintptr_t)a); };
    expect(range_holds(4096, 4096, at(4096), 4096), true, "the whole range");
    expect(range_holds(4096, 4096, at(8176), 16), true, "its last bytes");
    expect(range_holds(4096, 4096, at(8176), 17), false, "a byte beyond its end");
    expect(range_holds(4096, 4096, at(4096), 12288), false, "a range, a hole and another range");
    expect(range_holds(4096, 4096, at(4080), 16), false, "before it");
    expect(range_holds(4096, 4096, at(8192), 1), false, "behind it");
    expect(range_holds(4096, 4096, at(4096), ~(size_t)0), false, "more bytes than an address holds");
    expect(range_holds(~0ull - 4095, 4096, at(~0ull - 15), 16), true, "the end of the addresses");
    expect(range_holds(0, 0, at(4096), 1), false, "memory that is not known");
    if (argc > 1) {
        const size_t page = 4096;
        char* whole = nullptr;
        if (cudaFree(nullptr) != cudaSuccess || cudaHostAlloc(&whole, 8 * page, cudaHostAllocDefault) != cudaSuccess) return 100;
        expect(pinned_in_one_range(whole, 8 * page), true, "an allocation");
        expect(pinned_in_one_range(whole + 48, 5 * page), true, "a part of an allocation");
        char* const pages = static_cast<char*>(mmap(nullptr, 4 * page, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0));
        if (pages == MAP_FAILED) return 101;
        expect(pinned_in_one_range(pages, page), false, "pageable memory");
        if (cudaHostRegister(pages, page, cudaHostRegisterDefault) != cudaSuccess ||
            cudaHostRegister(pages + 2 * page, page, cudaHostRegisterDefault) != cudaSuccess) return 102;
        expect(pinned_in_one_range(pages, page), true, "a registration");
        expect(pinned_in_one_range(pages + 2 * page + 16, page - 16), true, "the end of a registration");
        expect(pinned_in_one_range(pages, 3 * page), false, "two registrations and the hole between them");
        expect(pinned_in_one_range(pages + 16, page), false, "past the end of a registration");
        void* device = nullptr;
        void* managed = nullptr;
        if (cudaMalloc(&device, page) != cudaSuccess || cudaMallocManaged(&managed, page) != cudaSuccess) return 103;
        expect(pinned_in_one_range(device, 16), false, "device memory");
        expect(pinned_in_one_range(managed, 16), false, "managed memory");
        expect(cudaGetLastError() == cudaSuccess, true, "no error is left behind");
        cudaFree(device);
        cudaFree(managed);
        cudaHostUnregister(pages);
        cudaHostUnregister(pages + 2 * page);
        munmap(pages, 4 * page);
        cudaFreeHost(whole);
    }
    printf("%d wrong\n", bad);
    return bad;
}
