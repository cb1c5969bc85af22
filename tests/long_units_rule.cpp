// Which instance runs a whole step: reads "precision log2(block) long_tiles other_tiles other_ragged" a line, writes 0 or 1.
#include <cstdio>

#include "ciera_internal.cuh"

int main() {
    int dtype;
    unsigned log2b;
    unsigned long long longs, others, ragged;
    while (scanf("%d %u %llu %llu %llu", &dtype, &log2b, &longs, &others, &ragged) == 5)
        printf("%d\n", ciera::runs_as_long_units(dtype, log2b, longs, others, ragged) ? 1 : 0);
    return 0;
}
