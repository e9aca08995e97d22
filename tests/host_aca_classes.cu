// Host harness of the ACA launch classes (csrc/hbi_internal.h): prints "<tau> <sig> <class> <class when
// stepwise>" for block shapes from single elements to a leaf against the largest clusters.
#include <cstdio>

#include "../paper_2110_12165_gb300/csrc/hbi_internal.h"

using namespace hbi;

int main() {
    const int sizes[] = {1, 2, 16, 20, 21, 40, 41, 64, 65, 127, 128, 129, 256, 4000, 60000, 1000000};
    for (int tau : sizes)
        for (int sig : sizes) printf("%d %d %d %d\n", tau, sig, aca_class(tau, sig, false), aca_class(tau, sig, true));
    return 0;
}
