// Host check of load_pair: with `two` false it touches one value only.  The value is the last one before a page that cannot be
// read, so a read of the next one ends the program with a signal.
#include <stdio.h>
#include <sys/mman.h>
#include <unistd.h>

#include "../../paper_1602_05700_gb300/csrc/lap_int.cuh"

int main() {
    const long page = sysconf(_SC_PAGESIZE);
    char* m = (char*)mmap(nullptr, 2 * page, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    if (m == MAP_FAILED || mprotect(m + page, page, PROT_NONE)) return 2;
    double* last = (double*)(m + page) - 1;
    last[-1] = 3.0;
    last[0] = 5.0;
    double a[2], b[2];
    hg::load_pair(last - 1, true, a);
    hg::load_pair(last, false, b);
    printf("%g %g %g %g\n", a[0], a[1], b[0], b[1]);
    return 0;
}
