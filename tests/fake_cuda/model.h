// What the kernels do that the fake runtime models.
#pragma once
#include <functional>
#include <string>

// The kernel's work (by its mangled name), with its arguments read now.
std::function<void()> body(const std::string& kernel, void** args);
