// Rules that decide where a kernel may store, checked on the host (test
// infrastructure; built and run by tests/test_host_rules_cpu.py, no GPU needed).
// The argument names the group of checks.  Exit status 0 when all hold.
#include <cstdio>
#include <cstring>
#include <vector>

#include "conv_schedule.cuh"
#include "internal.h"

using namespace claire;

namespace {

int g_failures = 0;

void check(bool ok, const char* what)
{
    if (ok) return;
    std::printf("FAIL %s\n", what);
    ++g_failures;
}

// A result is formed in the caller's array only in memory that the context's GPU
// can store to.
void result_arrays()
{
    cudaPointerAttributes own{}, other{}, managed{}, host{};
    own.type = other.type = cudaMemoryTypeDevice;
    own.device = 1;
    other.device = 0;
    managed.type = cudaMemoryTypeManaged;
    host.type = cudaMemoryTypeHost;
    host.device = 1;
    auto at = [](size_t x) { return reinterpret_cast<const void*>(x); };
    const void *dst = at(0x10000), *in = at(0x90000);
    check(forms_in_place(own, 1, dst, 1000, in, 1000), "the context's GPU: in place");
    check(forms_in_place(managed, 1, dst, 1000, in, 1000), "managed memory: in place");
    check(!forms_in_place(other, 1, dst, 1000, in, 1000), "another GPU: by a copy");
    check(!forms_in_place(host, 1, dst, 1000, in, 1000), "host memory: by a copy");
    check(!forms_in_place(own, 1, at(0x10004), 1000, in, 1000), "off a 16-byte boundary: by a copy");
    check(!forms_in_place(own, 1, dst, 1000, at(0x10000 + 3996), 10), "one shared float behind: by a copy");
    check(forms_in_place(own, 1, dst, 1000, at(0x10000 + 4000), 10), "input right behind: in place");
    check(!forms_in_place(own, 1, dst, 1000, at(0x10000 - 36), 10), "one shared float in front: by a copy");
    check(forms_in_place(own, 1, dst, 1000, nullptr, 0), "no input: in place");
}

// The box of a scatter tile holds every node that its points add to, whatever the
// displacements (clamped to 2^20 cells, either sign, so extents reach 2^21).
void scatter_boxes()
{
    constexpr int cap = 6976, m = 4;
    const int lim = 1 << 20;
    int e[3];
    auto fits = [&](int s1, int s2, int s3) {
        const int a[3] = {0, -5, 7}, z[3] = {s1, s2 - 5, s3 + 7};
        return scatter_box_fits(a, z, m, cap, e);
    };
    check(fits(3, 7, 31) && e[0] == 7 && e[1] == 11 && e[2] == 35, "tile at rest");
    check(fits(12, 12, 23) && e[0] * e[1] * e[2] == 6912, "box just below the cap");
    check(!fits(12, 12, 24), "box just above the cap");
    check(fits(0, 0, 432) && !fits(0, 0, 433), "long rows up to the cap");
    // spans whose product wraps past 63 bits, to a negative, a small or a zero value
    check(!fits(2 * lim, 2 * lim, 2 * lim), "2^21 on every axis");
    check(!fits(2 * lim - 4, 2 * lim - 4, 2 * lim - 4), "extents 2^21: product 2^63");
    check(!fits((1 << 22) - 4, (1 << 21) - 4, (1 << 21) - 4), "product 2^64");
    for (int s1 : {0, 40, lim, 2 * lim})
        for (int s2 : {0, 40, lim, 2 * lim})
            for (int s3 : {0, 40, lim, 2 * lim}) {
                const bool want = (s1 + 4.0) * (s2 + 4.0) * (s3 + 4.0) <= cap;
                check(fits(s1, s2, s3) == want, "span grid");
            }
}

// The stacked convolution: between two waits, MMAs that touch the same columns have
// the same first column and the same width (only their order is defined); every
// output plane gets its depth taps 0, 1, 2 in that order.
void conv_schedule()
{
    struct Acc {
        int z0, nz;
    };
    for (int bdc : {1, 2, 4, 8}) {
        std::vector<int> next(bdc, 0);
        std::vector<Acc> open;  // issued and not waited for
        for (int sd = 0; sd < bdc + 2; ++sd) {
            if (stacked_wait(bdc, sd)) open.clear();
            const StackedPlane p = stacked_plane(bdc, sd);
            check(p.z0 >= 0 && p.nz >= 1 && p.nz <= 3 && p.z0 + p.nz <= bdc, "columns of the brick");
            for (const Acc& a : open) {
                const bool overlap = p.z0 < a.z0 + a.nz && a.z0 < p.z0 + p.nz;
                check(!overlap || (p.z0 == a.z0 && p.nz == a.nz), "overlapping MMAs of different shapes");
            }
            open.push_back({p.z0, p.nz});
            for (int z = p.z0; z < p.z0 + p.nz; ++z) check(sd - z == next[z]++, "depth taps in order");
        }
        for (int z = 0; z < bdc; ++z) check(next[z] == 3, "three depth taps");
    }
}

}  // namespace

int main(int argc, char** argv)
{
    const char* group = argc > 1 ? argv[1] : "";
    if (!std::strcmp(group, "result_arrays"))
        result_arrays();
    else if (!std::strcmp(group, "scatter_boxes"))
        scatter_boxes();
    else if (!std::strcmp(group, "conv_schedule"))
        conv_schedule();
    else
        check(false, "unknown group");
    if (!g_failures) std::printf("OK\n");
    return g_failures ? 1 : 0;
}
