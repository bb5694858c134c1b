// Controls of the runtime in fake_cudart.cpp.
#pragma once

#include <cstddef>
#include <functional>
#include <string>

void fake_fail_alloc(long k);  // the k-th device allocation from now on fails, once (-1: none)
long fake_allocs();            // device allocations since fake_fail_alloc
// launches on a non-blocking stream while a copy or set on the legacy stream
// was still to run, and the first such kernel's name
long fake_unordered(std::string *first);
void fake_on_launch(const char *name, std::function<void()> f);  // when such a kernel's turn comes
// at the launch of such a kernel, with its arguments; what it returns runs when its turn comes
void fake_on_launch_args(const char *name, std::function<std::function<void()>(void **)> f);
void fake_fail_pinned(bool fail);  // page-locked host memory
void fake_fail_launch(const char *name);  // launches of such kernels fail ("": none)
long fake_launches(const char *name);  // of kernels whose name contains the text
size_t fake_device_bytes();
size_t fake_uploaded();        // bytes copied from the host so far
void fake_settle();            // every queue runs
