// Host build of the rule on copies out (hd_internal.cuh) for tests/test_host_copy.py.
#include "../../paper_1402_1720_gb300/csrc/hd_internal.cuh"

extern "C" int hx_copy_by_kernel(unsigned long long dst, unsigned long long src, unsigned long long bytes)
{
    return hd::copy_by_kernel(reinterpret_cast<const void *>(dst), reinterpret_cast<const void *>(src),
                              bytes) ? 1 : 0;
}
