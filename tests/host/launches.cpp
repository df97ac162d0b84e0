// Launches as the host code issues them: the library's own objects, linked with a
// CUDA runtime that keeps device memory on the heap and records each launch.
//   slab Lx Ly Lz shape  a handle whose parameters change between sweeps; a line
//                        per slab launch: its CTAs per cluster, form, shared
//                        memory and threads, and what the descriptor it would
//                        read needs
//   tune Lx Ly Lz        the shapes AUTO takes: untuned, tuned (every candidate
//                        taking no time, so that the first one wins), with a bulk
//                        field, and without it again
//   auto Lx Ly Lz every  the shape AUTO takes without a measurement
//   film Lx Ly Lz shape H  a sweep of a handle; a line per launch: its form, and the
//                        rows of a packed word
//   thin items thick H   half-sweeps of eight films of 128x512x16 and, if thick, one
//                        of 120x240x1600; printed like grid's
//   pack n               the rows per word of n of each of the line-tension set's
//                        sizes in one set
//   grid items H0 H1 H2  half-sweeps of a set of a small, a medium and a large film
//                        in those bulk fields; a line per launch: its grid, the
//                        entries of the owner table, and its form
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

#include "ising_host.h"

namespace {
std::map<const void*, std::string> g_names;
bool g_quiet = false;
uint32_t g_blocks = 0;  // owner table entries of the film set in use
}

extern "C" {
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
  g_names[host] = name;
}
void** __cudaRegisterFatBinary(void*) { static void* h[4]; return h; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = calloc(n, 1); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {  // a GB300's
  *v = a == cudaDevAttrMaxSharedMemoryPerMultiprocessor ? 228 * 1024 : a == cudaDevAttrReservedSharedMemoryPerBlock ? 1024 : 152;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  memset(a, 0, sizeof *a);
  a->sharedSizeBytes = 1024;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 4;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = 10;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  if (g_quiet) return cudaSuccess;
  const std::string& name = g_names[f];
  // the last template argument of either update kernel
  auto form = [&name](const char* kernel) {
    const size_t k = name.find(kernel);
    return k == std::string::npos ? -1 : atoi(name.c_str() + name.find("EE", k) - 1);
  };
  if (form("update_kernelI") >= 0) printf("grid %u blocks %u form %d\n", c->gridDim.x, g_blocks, form("update_kernelI"));
  const size_t film = name.find("update_film_kernelILi");
  if (film != std::string::npos)
    printf("form %d rows %d\n", form("update_film_kernelI"), atoi(name.c_str() + film + strlen("update_film_kernelILi")));
  const size_t at = name.find("slab_kernelILb");
  if (at == std::string::npos) return cudaSuccess;
  const bool tasks = name[at + strlen("slab_kernelILb1ELb")] == '1';
  uint32_t C = 1;
  for (unsigned i = 0; i < c->numAttrs; i++)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) C = c->attrs[i].val.clusterDim.x;
  const isg::FilmDesc& d = **static_cast<isg::FilmDesc**>(args[0]);
  printf("C %u tasks %d fit %d smem %zu need %u threads %u want %u\n", C, tasks, isg::slab_tasks_fit(d, C),
         (size_t)c->dynamicSmemBytes, isg::slab_dyn_bytes(d, C, tasks), c->blockDim.x,
         isg::cluster_threads(d, C, 1, tasks));
  return cudaSuccess;
}
// calls that need do nothing here
#define NOTHING(name)              \
  int nothing_##name() asm(#name); \
  int nothing_##name() { return 0; }
NOTHING(__cudaGetKernel) NOTHING(__cudaLaunchKernel) NOTHING(__cudaPopCallConfiguration)
NOTHING(__cudaPushCallConfiguration) NOTHING(__cudaRegisterFatBinaryEnd) NOTHING(__cudaRegisterVar)
NOTHING(__cudaUnregisterFatBinary) NOTHING(cudaEventCreate) NOTHING(cudaEventCreateWithFlags) NOTHING(cudaEventDestroy)
NOTHING(cudaEventElapsedTime) NOTHING(cudaEventQuery) NOTHING(cudaEventRecord) NOTHING(cudaEventSynchronize)
NOTHING(cudaFreeHost) NOTHING(cudaFuncSetAttribute) NOTHING(cudaGetLastError) NOTHING(cudaGetSymbolAddress)
NOTHING(cudaMemcpy) NOTHING(cudaMemcpyFromSymbol) NOTHING(cudaSetDevice) NOTHING(cudaStreamCreateWithFlags)
NOTHING(cudaStreamDestroy) NOTHING(cudaStreamQuery) NOTHING(cudaStreamSynchronize) NOTHING(cudaStreamWaitEvent)
}

namespace {
void ok(int rc) {
  if (rc) { printf("status %d: %s\n", rc, ising_last_error()); exit(1); }
}

// two sweeps of a film set
struct Size {
  int Lx, Ly, Lz;
  double H;
};
void set(uint32_t items, const std::vector<Size>& films) {
  isg::FilmSet fs;
  fs.items = items;
  fs.h.resize(films.size());
  for (size_t i = 0; i < films.size(); i++) {
    memset(&fs.h[i], 0, sizeof fs.h[i]);
    isg::fill_geometry(fs.h[i], films[i].Lx, films[i].Ly, films[i].Lz, ISING_Y_GAPBC, ISING_X_FREE, 1, (uint32_t)i);
    isg::build_tables(fs.h[i], 1.0, films[i].H, 0.5, 3.0);
  }
  ok(fs.init_device());
  fs.layout();
  ok(fs.upload());
  g_blocks = fs.hh.upd_blocks;
  if (g_quiet)
    for (const auto& d : fs.h) printf("rows %u\n", d.pack);
  ok(fs.enqueue_sweeps(0, 2));
}

void tune(ising* h) {
  auto show = [h] {
    int s = 0;
    ok(ising_get_shape(h, 1, &s));
    printf("shape %d\n", s);
  };
  show();
  ok(ising_autotune(h, 1, nullptr));
  show();
  ok(ising_set_options(h, ISING_Y_GAPBC, ISING_X_FREE, 0.3, 0));
  show();
  ok(ising_set_options(h, ISING_Y_GAPBC, ISING_X_FREE, 0.0, 0));
  show();
  ok(ising_destroy(h));
}
}  // namespace

// slab: sweeps at J = 1, H = 0, then J = -1, J = 1, H = 0.3, H = 0
int main(int, char** a) {
  if (!strcmp(*++a, "grid")) {
    set((uint32_t)atoi(a[1]), {{4, 6, 8, atof(a[2])}, {24, 30, 96, atof(a[3])}, {120, 240, 1600, atof(a[4])}});
    return 0;
  }
  if (!strcmp(*a, "pack")) {
    std::vector<Size> films;
    for (int i = 0; i < atoi(a[1]); i++)
      for (int z : {16, 32, 48, 64, 96}) films.push_back({1536 / z, 9216 / z, z, 0.0});
    g_quiet = true;
    set(1, films);
    return 0;
  }
  if (!strcmp(*a, "thin")) {
    std::vector<Size> films(8, Size{128, 512, 16, atof(a[3])});
    if (atoi(a[2])) films.push_back({120, 240, 1600, 0.0});
    set((uint32_t)atoi(a[1]), films);
    return 0;
  }
  ising* h = nullptr;
  ok(ising_create(atoi(a[1]), atoi(a[2]), atoi(a[3]), 1.0, 0.5, 3.0, 1, &h));
  if (!strcmp(a[0], "auto")) {
    int s = 0;
    ok(ising_get_shape(h, (uint32_t)atoi(a[4]), &s));
    printf("shape %d\n", s);
    ok(ising_destroy(h));
    return 0;
  }
  if (!strcmp(a[0], "tune")) {
    g_quiet = true;
    tune(h);
    return 0;
  }
  ok(ising_set_shape(h, atoi(a[4])));
  if (!strcmp(a[0], "film")) {
    ok(ising_set_options(h, ISING_Y_GAPBC, ISING_X_FREE, atof(a[5]), 0));
    ok(ising_sweep(h, 1, 1));
    ok(ising_destroy(h));
    return 0;
  }
  ok(ising_sweep(h, 2, 1));
  ok(ising_set_params(h, -1.0, 0.5, 3.0));
  ok(ising_sweep(h, 2, 1));
  ok(ising_set_params(h, 1.0, 0.5, 3.0));
  ok(ising_sweep(h, 2, 1));
  ok(ising_set_options(h, ISING_Y_GAPBC, ISING_X_FREE, 0.3, 0));
  ok(ising_sweep(h, 2, 1));
  ok(ising_set_options(h, ISING_Y_GAPBC, ISING_X_FREE, 0.0, 0));
  ok(ising_sweep(h, 2, 1));
  ok(ising_destroy(h));
  return 0;
}
