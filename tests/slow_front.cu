// A kernel that lets the next one on its stream start at once and then takes its time (a bounded one).
#include <cstdint>

__global__ void slow_front_kernel(unsigned long long ns) {
    asm volatile("griddepcontrol.launch_dependents;");
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    do {
        __nanosleep(1000);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    } while (t - t0 < ns);
}
extern "C" int slow_front(unsigned long long ns, void* stream) {
    slow_front_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(ns < 3000000000ull ? ns : 3000000000ull);
    return (int)cudaGetLastError();
}
