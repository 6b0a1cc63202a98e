// Row lists of the N = 2^16 transform kernels: the rows of one kind (arithmetic) inside a period of `period` rows.
// Launch row y covers buffer row (y / count) * period + row[y % count] on prime[y % count].
#pragma once
#include <stdint.h>
struct RowList {
    uint32_t period, count;
    uint8_t row[252], prime[252];
};
