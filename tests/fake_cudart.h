// A stand-in for the CUDA runtime that runs nothing: "device" memory is host
// memory, copies are copies, kernels are counted by name and do no work.  It keeps
// the order of streams: which ones have work queued since they were last waited
// for, whether a stream-ordered buffer is returned in the order of another stream
// while its own still has some, and whether a stream works beside a graph that was
// captured from its work and runs on another stream.  Allocations and kernels can
// be made to fail.  For tests of the library's host code without a GPU (link the library's
// objects with fake_cudart.cpp instead of the runtime).
#pragma once
#include <cstddef>

namespace fake {
extern int violations;           // buffers returned too early or by the wrong call, streams that race
extern bool capture;             // whether streams can be captured
extern int fail_alloc_at;        // the n-th allocation from now fails (0: none)
extern std::size_t fail_over;    // device allocations of more bytes fail (0: none)
extern const char* fail_kernel;  // the next kernel whose name contains this fails
std::size_t live();              // buffers not given back
std::size_t held();              // their bytes
int waits();                     // streams made to wait for another one's event
int launched(const char* name);  // kernels so far whose name contains `name`
}  // namespace fake
