// Thread-local error message plumbing shared by the host parts of libqe.
#pragma once
#include <cstdarg>
#include <cstdint>
#include <new>

namespace qe {
// Records a formatted message for qe_last_error() and returns `status` unchanged.
int32_t fail(int32_t status, const char* fmt, ...);
void clear_error();
int32_t out_of_memory();  // the status of a call that could not allocate host memory
}  // namespace qe

// Ends an entry point written as a function-try-block: no exception leaves the C interface.
#define QE_NO_MEMORY \
  catch (const std::bad_alloc&) { return qe::out_of_memory(); }
