// Host run of the rule that chooses the sweep kernel (pv_batch.cuh): reads pairs
// "tiles SMs" from stdin, prints the FP32 and the FP64 mode of each.
#include <cstdio>

#include "pv_batch.cuh"

int main() {
    int tiles, sms;
    while (scanf("%d %d", &tiles, &sms) == 2)
        printf("%d %d\n", (int)pv::sweep_mode<float>(tiles, sms), (int)pv::sweep_mode<double>(tiles, sms));
    return 0;
}
