/* A CUDA runtime that runs nothing: it records the launches the library
 * makes (kernel name, grid, block, shared memory), so that the host side's
 * choices can be tested without a GPU.  Loaded before the library, its
 * symbols stand in front of libcudart's.  Occupancy is what 2048 threads, 32
 * CTAs and 228 KB of shared memory an SM allow; times and stream states are
 * set by the test. */
#include <stddef.h>
#include <stdint.h>
#include <string.h>
#include <time.h>

#define MAXL (1 << 19)
typedef struct { unsigned x, y, z; } dim3_t;
typedef struct { char name[256]; unsigned grid, block; uint64_t smem; } launch_t;

static struct { const void* host; char name[256]; } g_fn[512];
static int g_nfn;
static launch_t g_launch[MAXL];
static int g_nlaunch;
static double g_ready_s;   /* the stream is busy until this monotonic time */
static float g_elapsed_ms = 1.0f;
static struct { dim3_t grid, block; size_t smem; void* stream; } g_conf;

static double now_s(void) {
    struct timespec t;
    clock_gettime(CLOCK_MONOTONIC, &t);
    return (double)t.tv_sec + 1e-9 * (double)t.tv_nsec;
}

/* ---- for the tests ---- */
int fake_launches(void) { return g_nlaunch; }
const launch_t* fake_launch(int i) { return &g_launch[i]; }
void fake_reset(void) { g_nlaunch = 0; }
void fake_busy_us(double us) { g_ready_s = now_s() + 1e-6 * us; }
void fake_elapsed_ms(float ms) { g_elapsed_ms = ms; }

/* ---- registration and launches ---- */
void** __cudaRegisterFatBinary(void* p) { static void* h; (void)p; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void** h, char* var, char* addr, const char* name, int ext, size_t n, int c, int g) {
    (void)h; (void)var; (void)addr; (void)name; (void)ext; (void)n; (void)c; (void)g;
}
void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* name, int lim, void* tid, void* bid,
                            void* bd, void* gd, int* ws) {
    (void)h; (void)dev; (void)lim; (void)tid; (void)bid; (void)bd; (void)gd; (void)ws;
    if (g_nfn < 512) {
        g_fn[g_nfn].host = host;
        strncpy(g_fn[g_nfn++].name, name, 255);
    }
}
unsigned __cudaPushCallConfiguration(dim3_t g, dim3_t b, size_t smem, void* st) {
    g_conf.grid = g;
    g_conf.block = b;
    g_conf.smem = smem;
    g_conf.stream = st;
    return 0;
}
int __cudaPopCallConfiguration(dim3_t* g, dim3_t* b, size_t* smem, void* st) {
    *g = g_conf.grid;
    *b = g_conf.block;
    *smem = g_conf.smem;
    *(void**)st = g_conf.stream;
    return 0;
}
int __cudaGetKernel(void** k, const void* host) { *k = (void*)host; return 0; }
int cudaLaunchKernel(const void* fn, dim3_t g, dim3_t b, void** args, size_t smem, void* st) {
    (void)args;
    (void)st;
    if (g_nlaunch < MAXL) {
        launch_t* l = &g_launch[g_nlaunch++];
        strcpy(l->name, "?");
        for (int i = 0; i < g_nfn; ++i)
            if (g_fn[i].host == fn) strcpy(l->name, g_fn[i].name);
        l->grid = g.x;
        l->block = b.x;
        l->smem = smem;
    }
    return 0;
}
int __cudaLaunchKernel(void* k, dim3_t g, dim3_t b, void** args, size_t smem, void* st) {
    return cudaLaunchKernel(k, g, b, args, smem, st);
}

/* ---- queries ---- */
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaSetDevice(int d) { (void)d; return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int d) { (void)attr; (void)d; *v = 152; return 0; }
int cudaFuncSetAttribute(const void* f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
int cudaGetLastError(void) { return 0; }
const char* cudaGetErrorString(int e) { (void)e; return "fake"; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int threads, size_t smem) {
    (void)f;
    int a = 2048 / threads, b = (int)(228 * 1024 / (smem + 1024));
    *n = a < b ? a : b;
    if (*n > 32) *n = 32;
    return 0;
}

/* ---- memory, streams, events ---- */
int cudaMemcpy(void* d, const void* s, size_t n, int k) { (void)s; (void)k; memset(d, 0, n); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int k, void* st) { (void)d; (void)s; (void)n; (void)k; (void)st; return 0; }
int cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, int k, void* st) {
    (void)d; (void)dp; (void)s; (void)sp; (void)w; (void)h; (void)k; (void)st;
    return 0;
}
int cudaMemsetAsync(void* d, int v, size_t n, void* st) { (void)d; (void)v; (void)n; (void)st; return 0; }
int cudaStreamQuery(void* st) { (void)st; return now_s() < g_ready_s ? 600 : 0; /* cudaErrorNotReady */ }
int cudaStreamCreateWithFlags(void** st, unsigned f) { (void)f; *st = (void*)16; return 0; }
int cudaStreamDestroy(void* st) { (void)st; return 0; }
int cudaEventCreate(void** e) { *e = (void*)16; return 0; }
int cudaEventDestroy(void* e) { (void)e; return 0; }
int cudaEventRecord(void* e, void* st) { (void)e; (void)st; return 0; }
int cudaEventSynchronize(void* e) { (void)e; return 0; }
int cudaEventElapsedTime(float* ms, void* a, void* b) { (void)a; (void)b; *ms = g_elapsed_ms; return 0; }
int cudaGetSymbolAddress(void** p, const void* s) { (void)s; *p = (void*)4096; return 0; }
