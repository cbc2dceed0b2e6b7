// A stand-in for the parts of the CUDA runtime that the launch sites use, on
// the host alone: several devices, function attributes that belong to one of
// them, and launches that are refused, as the runtime refuses them, where the
// current device lacks the attributes they need.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>
#include <tuple>

namespace {
int device = 0;
std::map<std::tuple<int, const void*, int>, int> attrs;  // (device, function, attribute) -> value
constexpr int kSmem = 8, kNonPortable = 14;              // cudaFuncAttribute values used
int launches = 0, refused = 0;

int attr(const void* f, int a) {
    auto it = attrs.find({device, f, a});
    return it == attrs.end() ? 0 : it->second;
}
int launch(const void* f, size_t smem, unsigned cluster) {
    const bool ok = (smem <= 48 * 1024 || attr(f, kSmem) >= (int)smem) && (cluster <= 8 || attr(f, kNonPortable));
    ++launches;
    if (!ok) ++refused;
    return ok ? 0 : 1;
}
}  // namespace

struct Dim3 {
    unsigned x, y, z;
};
struct LaunchAttr {  // cudaLaunchAttribute: id, padding, value
    int id;
    char pad[4];
    Dim3 dim;
    char rest[64 - sizeof(Dim3)];
};
struct LaunchConfig {  // cudaLaunchConfig_t
    Dim3 grid, block;
    size_t smem;
    void* stream;
    LaunchAttr* attrs;
    unsigned n;
};

extern "C" {
void fake_set_device(int d) { device = d; }
void fake_counts(int* l, int* r) {
    *l = launches, *r = refused;
    launches = refused = 0;
}
int cudaGetDevice(int* d) { return *d = device, 0; }
int cudaDeviceGetAttribute(int* v, int, int) { return *v = 152, 0; }
int cudaGetLastError() { return 0; }
int cudaFuncSetAttribute(const void* f, int a, int v) { return attrs[{device, f, a}] = v, 0; }
// device 2 takes no cluster; elsewhere the launch must be possible
int cudaOccupancyMaxActiveClusters(int* n, const void* f, const LaunchConfig* c) {
    *n = device != 2 && attr(f, kSmem) >= (int)c->smem && attr(f, kNonPortable);
    return 0;
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int, size_t smem, unsigned) {
    return *n = attr(f, kSmem) >= (int)smem ? 2 : 0, 0;
}
int cudaLaunchKernelExC(const LaunchConfig* c, const void* f, void**) {
    unsigned cluster = 1;
    for (unsigned k = 0; k < c->n; ++k)
        if (c->attrs[k].id == 4) cluster = c->attrs[k].dim.x * c->attrs[k].dim.y * c->attrs[k].dim.z;
    return launch(f, c->smem, cluster);
}
// the <<< >>> form
static size_t pushed = 0;
unsigned __cudaPushCallConfiguration(Dim3, Dim3, size_t smem, void*) { return pushed = smem, 0; }
int __cudaPopCallConfiguration(Dim3* g, Dim3* b, size_t* smem, void** s) {
    memset(g, 0, sizeof *g), memset(b, 0, sizeof *b);
    return *smem = pushed, *s = nullptr, 0;
}
int __cudaGetKernel(const void** k, const void* f) { return *k = f, 0; }
int __cudaLaunchKernel(const void* k, Dim3, Dim3, void**, size_t smem, void*) { return launch(k, smem, 1); }
int cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long, int* q) {
    struct Fake {
        static int encode() { return 0; }  // cuTensorMapEncodeTiled; its arguments are the caller's
    };
    return *fn = (void*)&Fake::encode, *q = 0, 0;
}
void** __cudaRegisterFatBinary(void*) {
    static void* handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 1; }
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
}
