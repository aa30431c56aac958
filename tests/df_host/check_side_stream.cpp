// The second stream of a call (csrc/side_stream.cuh) against a CUDA runtime that only writes down
// what it is asked: on every way out the owner waits for the stream's work before it is released.
// Prints one word per case.
#include <cstdio>
#include <string>

#include "cuda_runtime.h"  // the fake, below the include path's first entry
#include "side_stream.cuh"

std::string fake_log;
int fake_fail = 0;  // which call fails: 'r' record, 'w' wait

using namespace egs;

int main()
{
    int a;
    cudaStream_t owner = (cudaStream_t)&a;
    {
        SideStream x;  // work left on it: an early return
        x.create(owner, true);
        fake_log.clear();
        x.open = true;
    }
    std::printf("early=%s\n", fake_log.c_str());
    fake_log.clear();
    {
        SideStream x;  // joined by the call itself: nothing twice
        x.create(owner, false);
        x.open = true;
        fake_log.clear();
        x.join();
        fake_log += '|';
    }
    std::printf("joined=%s\n", fake_log.c_str());
    for (char f : {'r', 'w'}) {
        SideStream x;
        x.create(owner, false);
        x.open = true;
        fake_log.clear();
        fake_fail = f;
        const bool bad = x.join() != cudaSuccess;
        fake_fail = 0;
        std::printf("fail_%c=%s%s\n", f, fake_log.c_str(), bad ? "!" : "");
    }
    fake_log.clear();
    { SideStream x; }  // never created
    std::printf("none=%s\n", fake_log.c_str());
    return 0;
}
