// What the kernels do that the fake runtime models.
#pragma once
#include <functional>
#include <string>

// The kernel's work (by its mangled name), with its arguments read now.
std::function<void()> body(const std::string& kernel, void** args);

// The runtime's side: whether p lies in a live allocation, and the record of what must not happen.
bool in_device_memory(const void* p);
void fault(const std::string& what);
