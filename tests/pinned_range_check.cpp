// The range check of pinned_range.cuh against a table of registrations that
// stands in for the driver's: prints "failures 0" when every answer is right.
#include <cstdio>

#include "pinned_range.cuh"

struct Range {
    uintptr_t start;
    size_t size;
};

int main() {
    // two registrations that touch, a gap, and one that ends with the address space
    const Range table[] = {{4096, 100}, {4196, 50}, {8192, 4096}, {UINTPTR_MAX - 9, 10}};
    auto query = [&](const void *p, uintptr_t *start, size_t *size) {
        for (const Range &r : table)
            if (reinterpret_cast<uintptr_t>(p) - r.start < r.size) {
                *start = r.start;
                *size = r.size;
                return true;
            }
        return false;
    };
    auto mapped_elsewhere = [&](const void *, uintptr_t *start, size_t *size) {
        *start = 1 << 20;
        *size = 4096;
        return true;
    };
    int failures = 0;
    auto expect = [&](uintptr_t at, int64_t bytes, bool want) {
        const bool got = cpt::in_one_range(reinterpret_cast<const void *>(at), bytes, query);
        if (got != want) {
            ++failures;
            printf("%llu + %lld: %d\n", (unsigned long long)at, (long long)bytes, (int)got);
        }
    };
    expect(4096, 100, true);
    expect(4096, 101, false);      // on into the next registration
    expect(4095, 1, false);
    expect(4195, 1, true);
    expect(4195, 2, false);
    expect(4196, 50, true);
    expect(4196, 51, false);       // past the end
    expect(8192 + 13, 4083, true);
    expect(8192 + 13, 4084, false);
    expect(8192, INT64_MAX, false);
    expect(8192, -1, false);
    expect(5000, 1, false);        // not pinned
    expect(UINTPTR_MAX - 9, 10, true);
    expect(UINTPTR_MAX - 5, 7, false);
    if (cpt::in_one_range(reinterpret_cast<const void *>(8192), 1, mapped_elsewhere)) ++failures;
    printf("failures %d\n", failures);
    return failures != 0;
}
