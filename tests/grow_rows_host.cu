// Host check of cq_grow_rows (cq_internal.cuh): a buffer that an allocator with a limit grows, as
// the learned start's do.  Reads row counts from stdin, the limit first; writes for each whether
// the call succeeded and the rows there is room for and memory of afterwards.  No GPU is involved.
#include <cstdio>

#include "../paper_2205_08941_gb300/csrc/cq_internal.cuh"

int main()
{
    long limit, rows, held = 0;  // rows of memory held
    int64_t have = 0;
    if (std::scanf("%ld", &limit) != 1) return 1;
    while (std::scanf("%ld", &rows) == 1) {
        const cq_status st = cq_grow_rows(have, rows, [&] {
            held = 0;  // as cq_alloc: the old memory goes first
            if (rows > limit) return CQ_ERR_NOMEM;
            held = rows;
            return CQ_OK;
        });
        std::printf("%d %ld %ld\n", st == CQ_OK, (long)have, held);
    }
    return 0;
}
