// The host code of the library (csrc/capi.cu, unchanged) on the stand-in CUDA runtime of
// cuda_runtime.h.  In the place of each kernel launch stands a check that every array it
// would touch lies within one live allocation of device memory, whole, and what the host
// code reads back: the neighbour counts and the totals.  A launch that fails a check is
// counted (host_counter "bad") and touches nothing.
#include <string.h>

#include <cstdlib>
#include <functional>
#include <map>
#include <string>
#include <vector>

#include <cuda_runtime.h>

void host_symbol(void* p, size_t bytes);
template <typename T>
cudaError_t cudaGetSymbolAddress(void** p, T& symbol)
{
    *p = (void*)&symbol;
    host_symbol(*p, sizeof symbol);
    return cudaSuccess;
}

#include "../../paper_2603_01234_gb300/csrc/capi.cu"

namespace {

struct Block {
    size_t bytes;
    cudaMemoryType type;
    int device = 0;
};
std::map<char*, Block> blocks;
// this many more allocations of device (page-locked) memory succeed, then one fails (-1: none)
long fail_in = -1, fail_host_in = -1;
int needR = 20, needA = 10;
std::map<std::string, long> counters;
std::map<const void*, long> copies;  // by their addresses

const std::pair<char* const, Block>* block_of(const void* p)
{
    auto it = blocks.upper_bound((char*)p);
    if (it == blocks.begin()) return nullptr;
    --it;
    return (char*)p < it->first + it->second.bytes ? &*it : nullptr;
}

// p[0 ... bytes) is what a kernel may touch
void reach(const char* what, const void* p, size_t bytes)
{
    const auto* b = p ? block_of(p) : nullptr;
    if (b && (const char*)p + bytes <= b->first + b->second.bytes && b->second.device == 0) return;
    ++counters["bad"];
    ++counters[std::string("bad ") + what];
}

}  // namespace

struct HostStream {
    HostGraph* capture = nullptr;
};
struct HostEvent {};
struct HostGraph {
    std::vector<std::function<void()>> ops;
};
struct HostGraphExec {
    std::vector<std::function<void()>> ops;
};

namespace {

cudaError_t enqueue(cudaStream_t st, std::function<void()> f)
{
    if (st && st->capture) st->capture->ops.push_back(std::move(f));
    else f();
    return cudaSuccess;
}

cudaError_t allocate(void** p, size_t bytes, cudaMemoryType type)
{
    const bool dev = type == cudaMemoryTypeDevice;
    long& f = dev ? fail_in : fail_host_in;
    if (f >= 0 && f-- == 0) return cudaErrorMemoryAllocation;
    char* q = (char*)aligned_alloc(256, (bytes + 255) / 256 * 256);
    memset(q, 0x5a, bytes);
    blocks[q] = {bytes, type};
    ++counters[dev ? "malloc" : "malloc_host"];
    *p = q;
    return cudaSuccess;
}

cudaError_t release(void* p)
{
    auto it = blocks.find((char*)p);
    if (it == blocks.end()) return cudaErrorInvalidValue;
    blocks.erase(it);
    free(p);
    return cudaSuccess;
}

}  // namespace

void host_symbol(void* p, size_t bytes) { blocks[(char*)p] = {bytes, cudaMemoryTypeDevice}; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { return allocate(p, n, cudaMemoryTypeDevice); }
cudaError_t cudaMallocHost(void** p, size_t n) { return allocate(p, n, cudaMemoryTypeHost); }
cudaError_t cudaFree(void* p) { return release(p); }
cudaError_t cudaFreeHost(void* p) { return release(p); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p)
{
    const auto* b = block_of(p);
    *a = {b ? b->second.type : cudaMemoryTypeUnregistered, b ? b->second.device : -1, (void*)p, (void*)p};
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t st) { return enqueue(st, [=] { memset(p, v, n); }); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind)
{
    ++copies[d];
    ++copies[s];
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st)
{
    ++copies[d];
    ++copies[s];
    return enqueue(st, [=] { memcpy(d, s, n); });
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t st)
{
    return enqueue(st, [=] { for (size_t k = 0; k < h; ++k) memcpy((char*)d + k * dp, (const char*)s + k * sp, w); });
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = new HostStream; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { delete s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) { s->capture = new HostGraph; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) { *g = s->capture; s->capture = nullptr; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long)
{
    ++counters["instantiate"];
    *e = new HostGraphExec{g->ops};
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t)
{
    ++counters["replay"];
    for (auto& f : e->ops) f();
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { delete e; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = new HostEvent; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = new HostEvent; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }

namespace nep {

template <typename real>
cudaError_t launch_cell_build(const PlanCounts* pc, int n_cap, int, int ncell_cap, bool zero_counts, bool, const WorkItem*,
                              const ReqInfo*, const ModelDesc<real>*, const double* pos, const int* types, int* cell_of,
                              PosRec<real>* rec_user, int* cell_count, int* cell_local, int* block_off, int* cell_fill,
                              int* perm_tmp, int* perm, int* cell_start, int* cell_s, PosRec<real>* rec_s, int* err,
                              cudaStream_t st)
{
    return enqueue(st, [=] {
        const size_t n = n_cap, nc = ncell_cap;
        reach("pos", pos, 24 * (size_t)pc->n), reach("types", types, 4 * (size_t)pc->n), reach("cell_of", cell_of, 4 * n);
        reach("rec", rec_user, sizeof(PosRec<real>) * n), reach("rec_s", rec_s, sizeof(PosRec<real>) * n);
        reach("perm", perm, 4 * n), reach("perm_tmp", perm_tmp, 4 * n), reach("cell_s", cell_s, 4 * n);
        reach("cell_local", cell_local, 4 * nc), reach("cell_fill", cell_fill, 4 * nc), reach("cell_start", cell_start, 4 * (nc + 1));
        reach("err", err, 4), reach("cell_count", cell_count, 4 * nc), reach("block_off", block_off, 4 * (kScanItems + 1));
        if (counters["bad"]) return;
        for (int i = 0; i < n_cap; ++i) perm[i] = i, cell_s[i] = 0;
        if (zero_counts) return;
        // the counters a build starts from are zero; what the scan of a build leaves is zero too
        bool clear = block_off[kScanItems] == 0;
        for (size_t c = 0; c < nc; ++c) clear &= cell_count[c] == 0;
        if (!clear) ++counters["uncleared"];
    });
}

template <typename real>
cudaError_t launch_kick_drift_bin(const PlanCounts*, int, const WorkItem*, const ReqInfo*, const ModelDesc<real>*,
                                  const int*, const TypeTable&, int, double, double, double*, double*, const double*, int*,
                                  PosRec<real>*, int*, int*, cudaStream_t st)
{
    return enqueue(st, [] {});
}

template <typename real>
cudaError_t launch_neighbors(const NeighborArgs<real>& a, int, int, size_t, cudaStream_t st)
{
    return enqueue(st, [=] {
        const size_t n = a.n;
        reach("nlR", a.nlR, 4 * n * a.mnR), reach("nlA", a.nlA, 4 * n * a.mnA);
        reach("cntR", a.cntR, 4 * n), reach("cntA", a.cntA, 4 * n), reach("rec_s", a.rec, sizeof(PosRec<real>) * n);
        if (a.accF) reach("accF", a.accF, 32 * n);
        if (a.accW) reach("accW", a.accW, 96 * n);
        if (a.rec32) reach("rec32", a.rec32, 16 * n);
        if (counters["bad"]) return;
        memset(a.cntR, 0, 4 * n), memset(a.cntA, 0, 4 * n);
        a.maxcnt[0] = needR;
        a.maxcnt[1] = needA;
    });
}

template <typename real>
cudaError_t launch_evaluate(int, int, int, int, const EvalArgs<real>& a, int items_cap, bool, size_t, size_t,
                            cudaStream_t st, cudaEvent_t, int, int, int)
{
    ++counters["evaluate"];
    return enqueue(st, [=] {
        const size_t n = a.n;
        reach("nlR", a.nlR, 4 * n * a.mnR), reach("nlA", a.nlA, 4 * n * a.mnA), reach("U", a.U, sizeof(real) * n);
        reach("e", a.e, sizeof(real) * n * a.e_stride), reach("wsum", a.wsum, sizeof(real) * 9 * n);
        reach("partial", a.partial, 80 * (size_t)items_cap), reach("icounter", a.icounter, 4 * (size_t)items_cap);
        reach("force", a.force, 24 * (size_t)a.counts->n);
        if (sizeof(real) == 8) reach("fang", a.fang, 24 * n * a.mnA);
        else reach("accF", a.accF, 32 * n);
        const size_t nq = a.counts->n_req;
        reach("totals", a.totals, 80 * nq);
        if (a.counts->energy) reach("energy", a.counts->energy, 8 * nq);
        if (a.counts->virial) reach("virial_total", a.counts->virial, 72 * nq);
        if ((uintptr_t)a.counts->energy % 8 || (uintptr_t)a.counts->virial % 8) ++counters["bad"];
        if (counters["bad"]) return;
        for (size_t r = 0; r < nq; ++r)  // energy r + 0.5, virial component k r + k
            for (int t = 0; t < 10; ++t) write_total(a.counts->energy, a.counts->virial, a.totals, (int)r, t, (double)r + (t ? t - 1 : 0.5));
    });
}

template <typename real>
bool evaluate_shape_supported(int nR, int nA, int KR, int KA) { return nR == 5 && nA == 4 && KR == 8 && KA == 8; }
template <typename real>
cudaError_t evaluate_set_smem(int, int, int, int, size_t, size_t) { return cudaSuccess; }

cudaError_t launch_kick(int, const int*, const double*, int, double, double*, const double*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_sample(int, const int*, const double*, int, const double*, const double*, double*, unsigned int*, double*, int*, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_scale(int, double*, double, double, double, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_bussi(int, const int*, const double*, int, double*, double*, unsigned int*, const double*, int*, double, double, double, double*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_hnemd_force(int, const double*, const double*, const double*, double*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_heat(int, const int*, const double*, int, const double*, const double*, const double*, double*, unsigned int*, double*, double*, const int*, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_cg_map(int, int, const int*, const int*, const double*, const double*, const double*, const double*, const CellGrid&, int, double*, double*, double*, cudaStream_t) { return cudaSuccess; }

#define NEP_INSTANTIATE(real)                                                                                              \
    template cudaError_t launch_cell_build<real>(const PlanCounts*, int, int, int, bool, bool, const WorkItem*,            \
                                                 const ReqInfo*, const ModelDesc<real>*, const double*, const int*, int*, \
                                                 PosRec<real>*, int*, int*, int*, int*, int*, int*, int*, int*,           \
                                                 PosRec<real>*, int*, cudaStream_t);                                      \
    template cudaError_t launch_kick_drift_bin<real>(const PlanCounts*, int, const WorkItem*, const ReqInfo*,             \
                                                     const ModelDesc<real>*, const int*, const TypeTable&, int, double,   \
                                                     double, double*, double*, const double*, int*, PosRec<real>*, int*,  \
                                                     int*, cudaStream_t);                                                 \
    template cudaError_t launch_neighbors<real>(const NeighborArgs<real>&, int, int, size_t, cudaStream_t);               \
    template cudaError_t launch_evaluate<real>(int, int, int, int, const EvalArgs<real>&, int, bool, size_t, size_t,      \
                                               cudaStream_t, cudaEvent_t, int, int, int);                                 \
    template bool evaluate_shape_supported<real>(int, int, int, int);                                                     \
    template cudaError_t evaluate_set_smem<real>(int, int, int, int, size_t, size_t);
NEP_INSTANTIATE(float)
NEP_INSTANTIATE(double)

}  // namespace nep

extern "C" {
void host_set(const char* what, long value)
{
    const std::string w = what;
    if (w == "fail_in") fail_in = value;
    else if (w == "fail_host_in") fail_host_in = value;
    else if (w == "needR") needR = (int)value;
    else if (w == "needA") needA = (int)value;
}
// the rules of dispatch.h: the neighbour kernel of count boxes of n particles, and whether a batch
// runs the group kernels
int host_neighbor_form(int boxes, const int* n, const int* types, const double* box, const int* pbc, const double* rc,
                       int fp64)
{
    NeighborLoad w;
    for (int r = 0; r < boxes; ++r) {
        CellGrid g;
        if (make_grid(nullptr, rc[r], box + 3 * r, pbc + 3 * r, g) != NEP_OK) return -1;
        w.add(g, n[r], types[r]);
    }
    return neighbor_form(w, fp64 != 0);
}
int host_by_groups(int n, int items, int types, int hidden, int mnR, int mnA, int table_bytes, int virial, int fp64)
{
    return evaluate_by_groups({n, items, types, hidden, mnR, mnA, (size_t)table_bytes, virial != 0}, fp64 != 0);
}
// memory of the stand-in device (kind 2), of another device that kernels do not reach (3), or
// page-locked memory (1)
void* host_allocate(int kind, size_t bytes)
{
    void* p = nullptr;
    if ((kind == 1 ? cudaMallocHost(&p, bytes) : cudaMalloc(&p, bytes)) != cudaSuccess) return nullptr;
    if (kind == 3) blocks[(char*)p].device = 1;
    return p;
}
long host_counter(const char* what) { return counters[what]; }
long host_copies(const void* p) { return copies[p]; }
void host_reset_counters() { counters.clear(); }
}
