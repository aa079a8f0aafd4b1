/* A CUDA runtime of two devices for host code that launches kernels: nothing runs; a launch that asks for more dynamic shared memory than
 * its function has been allowed on the current device (48 KB, unless an attribute says more), or for more than 65,535 blocks along y or z, is
 * refused, as the real one does. */
#include <stddef.h>

enum { OK = 0, INVALID = 1, MAX_FN = 256 };
static int device, n_fn, launches;
static struct { const void* fn; int allowed[2]; } fns[MAX_FN];

static int* allowed(const void* fn) {
    for (int i = 0; i < n_fn; ++i)
        if (fns[i].fn == fn) return &fns[i].allowed[device];
    fns[n_fn].fn = fn;
    fns[n_fn].allowed[0] = fns[n_fn].allowed[1] = 48 * 1024;
    return &fns[n_fn++].allowed[device];
}

void fake_set_device(int d) { device = d; }
int fake_launches(void) { return launches; }

struct config { unsigned grid[3], block[3]; size_t smem; void* stream; void* attrs; unsigned n_attrs; };
int cudaLaunchKernelExC(const struct config* c, const void* fn, void** args) {
    if (c->smem > (size_t)*allowed(fn) || c->grid[1] > 65535 || c->grid[2] > 65535) return INVALID;
    ++launches;
    return OK;
}
int cudaFuncSetAttribute(const void* fn, int attr, int value) {
    if (attr == 8) *allowed(fn) = value;          /* cudaFuncAttributeMaxDynamicSharedMemorySize */
    return OK;
}
int cudaGetDevice(int* d) { *d = device; return OK; }
int cudaGetLastError(void) { return OK; }
void** __cudaRegisterFatBinary(void* p) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) {}
void __cudaUnregisterFatBinary(void** h) {}
void __cudaRegisterFunction(void** h, const char* f, char* d, const char* n, int l, void* a, void* b, void* c, void* e, int* w) {}

int cudaDeviceGetAttribute(int* v, int attr, int d) { *v = 148; return OK; }
static int encode_tiled(void) { return OK; }
int cudaGetDriverEntryPoint(const char* name, void** fn, unsigned long long flags, int* found) { *fn = (void*)encode_tiled; *found = 0; return OK; }
size_t _ZN3edg17step_region_wordsERK14edg_layer_desc(const void* d) { return 0; }     /* (edg_step.cu, which is not part of this) */
