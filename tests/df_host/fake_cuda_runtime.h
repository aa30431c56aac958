// A CUDA runtime for check_side_stream.cpp: every call appends a letter to fake_log (r record,
// w wait, y synchronise, s destroy stream, e destroy event); the one named by fake_fail fails.
#pragma once
#include <string>

typedef struct fake_stream *cudaStream_t;
typedef struct fake_event *cudaEvent_t;
typedef int cudaError_t;
enum { cudaSuccess = 0, cudaStreamNonBlocking = 1, cudaEventDisableTiming = 2 };
extern std::string fake_log;
extern int fake_fail;

inline cudaError_t fake_call(char c)
{
    fake_log += c;
    return fake_fail == c ? 1 : cudaSuccess;
}
inline cudaError_t cudaDeviceGetStreamPriorityRange(int *l, int *g)
{
    *l = 0;
    *g = -1;
    return cudaSuccess;
}
inline cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, int, int)
{
    static int one;
    *s = (cudaStream_t)&one;
    return cudaSuccess;
}
inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, int)
{
    static int one;
    *e = (cudaEvent_t)&one;
    return cudaSuccess;
}
inline cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return fake_call('r'); }
inline cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, int) { return fake_call('w'); }
inline cudaError_t cudaStreamSynchronize(cudaStream_t) { return fake_call('y'); }
inline cudaError_t cudaStreamDestroy(cudaStream_t) { return fake_call('s'); }
inline cudaError_t cudaEventDestroy(cudaEvent_t) { return fake_call('e'); }
