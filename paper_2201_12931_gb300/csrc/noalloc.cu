// Density filter without any allocation (see topo_filter_noalloc in topo.h).
//
// Some callers cannot allocate GPU memory at the point where they need the
// filter: a framework whose caching allocator already owns the device
// memory, or a loop that must not stall, since cudaMalloc and cudaFree can
// synchronise the whole device.  For them this file keeps the filter's
// scratch in one statically sized device array that every GPU loading the
// library holds until the process exits.
#include <mutex>
#include <string>

#include "common.cuh"

namespace topo {

namespace {

constexpr long long kNoAllocMaxElems = 1LL << 20;   // largest grid: 1,048,576 elements
constexpr int kNoAllocMaxDevices = 64;

// the tables of weight sums (filter_weights)
__device__ __align__(256) double g_filter_scratch[kFilterTables];

std::mutex g_mu;
double* g_scratch_ptr[kNoAllocMaxDevices] = {};
int g_nsm[kNoAllocMaxDevices] = {};

// device address of the scratch array and multiprocessors of the current
// device; looked up once per device with that device current
topo_status scratch_for_current_device(double** out, int* nsm, std::string* err) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) {
        *err = std::string("no usable CUDA device: ") + cudaGetErrorString(e);
        return TOPO_CUDA;
    }
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_scratch_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_filter_scratch);
        if (e != cudaSuccess || !p) {
            *err = std::string("cudaGetSymbolAddress of the filter scratch failed: ") + cudaGetErrorString(e);
            return TOPO_CUDA;
        }
        if (cudaDeviceGetAttribute(&g_nsm[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || g_nsm[dev] <= 0) {
            cudaGetLastError();
            g_nsm[dev] = 152;
        }
        g_scratch_ptr[dev] = static_cast<double*>(p);
    }
    *nsm = g_nsm[dev];
    *out = g_scratch_ptr[dev];
    return TOPO_OK;
}

}  // namespace

}  // namespace topo

using namespace topo;

extern "C" topo_status topo_filter_noalloc(int nx, int ny, int nz, double r, const double* in_dev,
                                           double* out_dev, int transpose, void* stream) {
    std::string err;
    auto fail = [&](topo_status st, const std::string& msg) {
        set_global_error(msg);
        return st;
    };
    if (nx <= 0 || ny <= 0 || nz <= 0) return fail(TOPO_BADARG, "grid dimensions must be positive");
    const long long ne = (long long)nx * ny * nz;
    if (ne > kNoAllocMaxElems)
        return fail(TOPO_BADARG, "grid has " + std::to_string(ne) +
                                     " elements; the no-allocation filter supports at most " +
                                     std::to_string(kNoAllocMaxElems));
    if (!(r > 0.0) || r > 6.0) return fail(TOPO_BADARG, "filter radius must be in (0, 6]");
    if (!in_dev || !out_dev || in_dev == out_dev) return fail(TOPO_BADARG, "bad pointers");
    double* scratch = nullptr;
    int nsm = 0;
    topo_status st = scratch_for_current_device(&scratch, &nsm, &err);
    if (st != TOPO_OK) return fail(st, err);
    long long launches = 0;
    const Ctx c{static_cast<cudaStream_t>(stream), &launches};
    Geom g;
    g.nx = nx;
    g.ny = ny;
    g.nz = nz;
    g.ne = ne;
    g.nn = (long long)(nx + 1) * (ny + 1) * (nz + 1);
    // the weights by class go to the kernels as an argument and the table of
    // weight sums is formed on the device, so no host memory is copied and
    // the launches depend on the arguments alone
    FilterPlan plan;
    filter_plan(g, r, nsm, false, &plan);
    plan.near[0] = plan.near[1] = plan.near[2] = plan.near[transpose ? 1 : 0];   // one table of weight sums
    filter_weights(c, g, plan, scratch);
    filter_launch(c, g, plan, transpose ? 1 : 0, in_dev, nullptr, 0.0, scratch, nullptr, out_dev);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(TOPO_CUDA, std::string("filter launch: ") + cudaGetErrorString(e));
    return TOPO_OK;
}
