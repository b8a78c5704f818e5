// Two kernels of a caller of the library, for tests of what its launches guarantee to their neighbours on the stream.
#include <cuda_runtime.h>

// Releases its dependents at once, works for `ns` nanoseconds and then writes *out = value.
__global__ void late_writer(int* out, int value, long long ns) {
    asm volatile("griddepcontrol.launch_dependents;");
    long long t0, t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    for (int i = 0; i < 1 << 20; ++i) {                  // (bounded whatever the timer says)
        __nanosleep(500);
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        if (t - t0 >= ns) break;
    }
    *out = value;
}

// Reads *in as soon as it is let run, without waiting for the kernel before it on the stream.
__global__ void early_reader(const int* in, int* seen) {
    *seen = __ldcg(in);
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

extern "C" __attribute__((visibility("default"))) int run_late_writer(int* out, int value, long long ns, void* stream) {
    late_writer<<<1, 1, 0, static_cast<cudaStream_t>(stream)>>>(out, value, ns);
    return (int)cudaGetLastError();
}

extern "C" __attribute__((visibility("default"))) int run_early_reader(const int* in, int* seen, void* stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(1);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, early_reader, in, seen);
}
