// Host build of the walk set-up's division (hd_geom.cuh) for tests/test_host_division.py.
#include "../../paper_1402_1720_gb300/csrc/hd_geom.cuh"

extern "C" int hx_fdiv32(long long a, int b, long long *rem)
{
    return hd::fdiv32(a, b, hd::rcp_int(b), *rem);
}
