// Memory for the pages of a host array that a copy is about to write.
#pragma once

#include <stddef.h>
#include <stdint.h>
#include <sys/mman.h>
#include <unistd.h>

#ifndef MADV_POPULATE_WRITE
#define MADV_POPULATE_WRITE 23
#endif

namespace ccz4 {

// Gives every page of [p, p + bytes) its memory, as a write to each would, by one request to the kernel, which
// changes no byte. Memory that cannot be written, or a kernel without the request (Linux before 5.14), is left as
// it is: whether the copy can write there is the copy's to say. (Touching the pages one by one ends the process
// where a page cannot be written.)
inline void populate_pages(void *p, size_t bytes) {
  const long size = sysconf(_SC_PAGESIZE);
  if (!p || bytes == 0 || size <= 0) return;
  const uintptr_t page = (uintptr_t)size, a = (uintptr_t)p / page * page, b = ((uintptr_t)p + bytes + page - 1) / page * page;
  (void)madvise((void *)a, b - a, MADV_POPULATE_WRITE);
}

}  // namespace ccz4
