// kernel_reaches for (memory type, device of the memory, device of the context):
// three integers per line in, 0 or 1 per line out.
#include <cstdio>

#include "lbm_reach.h"

int main() {
    int type, of, device;
    while (scanf("%d %d %d", &type, &of, &device) == 3) {
        cudaPointerAttributes a = {};
        a.type = (cudaMemoryType)type;
        a.device = of;
        printf("%d\n", lbmd::kernel_reaches(a, device) ? 1 : 0);
    }
    return 0;
}
