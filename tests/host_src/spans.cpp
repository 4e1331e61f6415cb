// Feeds sg::Spans the ranges on standard input ("+ start bytes" adds, "- start"
// removes) and prints 1 or 0 for each that was added or not.
#include <cstdio>

#include "../../paper_1706_04552_gb300/csrc/sg_spans.h"

int main()
{
    sg::Spans spans;
    char op;
    unsigned long long start, bytes;
    while (std::scanf(" %c %llu", &op, &start) == 2) {
        if (op == '-') {
            spans.remove((uintptr_t)start);
        } else if (std::scanf("%llu", &bytes) == 1) {
            std::printf("%d\n", (int)spans.add((uintptr_t)start, bytes));
        }
    }
    return 0;
}
