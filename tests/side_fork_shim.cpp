// The library's fork and join of side streams (SideFork, gsw_impl.cuh) over a
// stand-in for the three CUDA calls it makes, which logs them and fails one.
#include "gsw_impl.cuh"

namespace {
int calls, fail_at;            // the call that fails (counted from 1, 0: none)
bool forked[16], waited[16];   // per side stream: waits for the caller's, waited for

bool fails() { return ++calls == fail_at; }
int stream_of(cudaStream_t s) { return (int)(size_t)s - 100; }  // side streams are 100, 101, ..., events 200, 300, ...
int event_of(cudaEvent_t e) { return (int)(size_t)e - 300; }
bool recorded[16];
}  // namespace

extern "C" {

cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    if (fails()) return cudaErrorUnknown;
    if (event_of(e) >= 0 && stream_of(s) == event_of(e)) recorded[event_of(e)] = true;
    return cudaSuccess;
}

cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    if (fails()) return cudaErrorUnknown;
    if (event_of(e) < 0) forked[stream_of(s)] = true;
    else if (recorded[event_of(e)]) waited[event_of(e)] = true;
    return cudaSuccess;
}

cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    waited[stream_of(s)] = true;
    return cudaSuccess;
}

// Forks n streams, then a launch fails (leave) or all succeed and they are
// joined.  Returns the streams forked but not waited for; *made the calls made.
int sf_run(int n, int leave, int fail, int *made, int *status) {
    calls = 0;
    fail_at = fail;
    for (int k = 0; k < 16; k++) forked[k] = waited[k] = recorded[k] = false;
    gsw::SideStreams aux;
    for (int k = 0; k < gsw::kSideStreams; k++) {
        aux.s[k] = (cudaStream_t)(size_t)(100 + k);
        aux.join[k] = (cudaEvent_t)(size_t)(300 + k);
    }
    aux.fork = (cudaEvent_t)(size_t)200;
    *status = [&]() -> int {
        gsw::SideFork fork(aux, (cudaStream_t)(size_t)50);
        const cudaError_t e = fork.fork(n);
        if (e != cudaSuccess) return e;
        if (leave) return cudaErrorInvalidConfiguration;
        return fork.join();
    }();
    *made = calls;
    int open = 0;
    for (int k = 0; k < 16; k++) open += forked[k] && !waited[k];
    return open;
}

int sf_streams() { return gsw::kSideStreams; }

}  // extern "C"
