// Plays a step on host weights in parts against an object that only writes down what it is asked for:
//   host_step_order PARTS FAILING_CALL STICKY
// fails the call with that number (0 = none; STICKY = 1: and every copy after it) and prints what came, in order.
#include <stdio.h>
#include <stdlib.h>

#include "ciera_host_step.hpp"

struct Log {
    int failing, sticky, n = 0;
    int did(const char* what, int k) {
        ++n;
        const int rc = n == failing ? -100 - n : (sticky && failing && n > failing && what[0] == 'o') ? -1 : 0;
        printf("%s%d%s ", what, k, rc ? "!" : "");
        return rc;
    }
    int copy_in(uint32_t k) { return did("in", (int)k); }
    int step(uint32_t k) { return did("step", (int)k); }
    int copy_out(uint32_t k) { return did("out", (int)k); }
    void clear() { printf("clear "); }
    int join() { return did("join", 0); }
};

int main(int argc, char** argv) {
    if (argc != 4) return 2;
    Log log{atoi(argv[2]), atoi(argv[3])};
    const int rc = ciera::run_host_parts(log, (uint32_t)atoi(argv[1]));
    printf("rc%d\n", rc);
    return 0;
}
