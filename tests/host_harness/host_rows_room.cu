// Host build of the row passes' allocation rule (hd_rows.cuh) for tests/test_host_rows_room.py.
#include "../../paper_1402_1720_gb300/csrc/hd_rows.cuh"

// The walks allocated for n histories where `room` of them fit; *tries the attempts.
extern "C" long long hx_rows_room(long long n, long long room, int *tries)
{
    *tries = 0;
    long long last = 0;
    const long long got = hd::rows_walks_room(n, [&](int64_t walks) {
        ++*tries;
        last = walks;
        return walks <= room;
    });
    return got == 0 || got == last ? got : -1;
}
