// Rules that decide where a kernel may store, checked on the host (test
// infrastructure; built and run by tests/test_host_rules_cpu.py, no GPU needed).
// The argument names the group of checks.  Exit status 0 when all hold.
#include <cstdio>
#include <cstring>

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

}  // namespace

int main(int argc, char** argv)
{
    const char* group = argc > 1 ? argv[1] : "";
    if (!std::strcmp(group, "result_arrays"))
        result_arrays();
    else
        check(false, "unknown group");
    if (!g_failures) std::printf("OK\n");
    return g_failures ? 1 : 0;
}
