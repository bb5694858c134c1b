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
size_t fake_device_bytes();
size_t fake_uploaded();        // bytes copied from the host so far
void fake_settle();            // every queue runs
