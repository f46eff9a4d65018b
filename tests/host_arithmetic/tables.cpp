// table_reserve (lbm_host.h) against an allocator that fails on request.
#include "lbm_host.h"

#include <cstdlib>

namespace {
struct Record { long long a, b; };
Record* table = nullptr;
int cap = 0, live = 0, freed_before_alloc = 0;
bool fail = false, pending = false;
}  // namespace

extern "C" {

// Reserves n records (failing the allocation if asked); 1 if there is room.
int reserve(int n, int failing)
{
    fail = failing != 0;
    pending = false;
    return table_reserve(table, cap, (size_t)n,
                         [](size_t bytes) -> void* {
                             if (fail) return nullptr;
                             pending = true;
                             ++live;
                             return std::malloc(bytes);
                         },
                         [](void* p) {
                             freed_before_alloc += !pending;
                             --live;
                             std::free(p);
                         });
}
int capacity() { return cap; }
int buffers() { return live; }
int early_frees() { return freed_before_alloc; }
long long write_read(int n)   // the last record of n, through the table
{
    table[n - 1].b = n;
    return table[n - 1].b;
}

}  // extern "C"
