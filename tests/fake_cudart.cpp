// A CUDA runtime that launches nothing: the library's objects are linked against it, so that the host side (which kernel takes a
// call, with which grid, and what a failing query leaves behind) runs without a GPU.  Launches are recorded in order.
#include <map>
#include <string>
#include <vector>

#include <cuda_runtime_api.h>

struct Launch { std::string name; int ctas, cluster, smem, last; };
static std::map<const void *, std::string> &names() { static std::map<const void *, std::string> n; return n; }
static std::vector<Launch> launches;
static cudaError_t last_error = cudaSuccess;
static int cluster_answer[17], fail_queries = 0;

static void record(const void *func, dim3 grid, int cluster, size_t smem, int last) {
    launches.push_back(Launch{names()[func], (int)(grid.x * grid.y * grid.z), cluster, (int)smem, last});
}

extern "C" {
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, void *, void *, void *, void *, int *) { names()[host] = name; }
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
static dim3 c_grid, c_block; static size_t c_smem; static void *c_stream;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void *st) { c_grid = g; c_block = b; c_smem = s; c_stream = st; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *st) { *g = c_grid; *b = c_block; *s = c_smem; *(void **)st = c_stream; return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void *f, dim3 g, dim3, void **, size_t s, cudaStream_t) { record(f, g, 1, s, 0); return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
    int cluster = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.x;
    const bool batch = names()[f].find("score_select_batch_kernel") != std::string::npos;
    record(f, c->gridDim, cluster, c->dynamicSmemBytes, batch ? *(const bool *)args[21] : 0);   // its last argument: table staged
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { const cudaError_t e = last_error; last_error = cudaSuccess; return e; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *c) {
    if (fail_queries) return last_error = cudaErrorUnknown;
    *n = cluster_answer[c->attrs[0].val.clusterDim.x];
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t smem, unsigned) {
    if (fail_queries) return last_error = cudaErrorUnknown;
    *n = smem ? (int)(227 * 1024 / (smem + 1024)) : 6;
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *, const void *) { return last_error = cudaErrorInvalidValue; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return last_error = cudaErrorInvalidSymbol; }
cudaError_t cudaGetDriverEntryPoint(const char *, void **, unsigned long long, cudaDriverEntryPointQueryResult *) { return last_error = cudaErrorNotSupported; }

void fake_answers(int of1, int of2, int of4, int of8) { cluster_answer[1] = of1; cluster_answer[2] = of2; cluster_answer[4] = of4; cluster_answer[8] = of8; }
void fake_fail_queries(int fail) { fail_queries = fail; }
void fake_clear(void) { launches.clear(); last_error = cudaSuccess; }
int fake_launches(void) { return (int)launches.size(); }
const char *fake_launch(int i, int *ctas, int *cluster, int *smem, int *last) {
    const Launch &l = launches[i];
    *ctas = l.ctas; *cluster = l.cluster; *smem = l.smem; *last = l.last;
    return l.name.c_str();
}
}
