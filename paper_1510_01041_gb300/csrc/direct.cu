// direct.cu -- which fits the one-kernel branch-and-bound (direct.cuh) takes,
// its memory and its launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "direct.cuh"

namespace lms {
namespace direct {

// Whether the current device can hold one cluster of this kernel (16 CTAs are
// more than every device or partition of one grants), asked once per device,
// kernel and size of shared memory.
bool cluster_fits(const void *kern, const cudaLaunchConfig_t &cfg)
{
    static std::mutex mu;
    static std::map<std::tuple<int, const void *, size_t>, bool> known;
    int dev;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    std::lock_guard<std::mutex> lock(mu);
    const auto key = std::make_tuple(dev, kern, cfg.dynamicSmemBytes);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    int clusters = 0;
    const bool fits = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) == cudaSuccess && clusters > 0;
    if (known.size() > 4096) known.clear();
    known[key] = fits;
    return fits;
}

}  // namespace direct

using namespace direct;

namespace {

struct Single {
    int variant;
    TeamShape shape;
    size_t smem;
};

Single single_of(int n)
{
    Single s{};
    s.variant = n <= 2048 ? 0 : n <= 16384 ? 1 : 2;
    const int C = 16;
    if (s.variant == 0) {
        s.shape = Small::team(n, C, 4096, 256.0f);
        s.smem = Small::smem(n, 4096);
    } else if (s.variant == 1) {
        s.shape = Mid::team(n, C, 4096, 512.0f);
        s.smem = Mid::smem(n, 4096);
    } else {
        s.shape = Large::team(n, C, 4096, 1024.0f);
        s.smem = Large::smem(n, 4096);
    }
    return s;
}

Single float_single_of(int n)
{
    Single s{};
    s.variant = n <= 2048 ? 0 : 1;
    const int C = 16;
    if (s.variant == 0) {
        s.shape = FloatSmall::team(n, C, 4096, 256.0f);
        s.smem = FloatSmall::smem(n, 4096);
    } else {
        s.shape = FloatMid::team(n, C, 16384, 256.0f);
        s.smem = FloatMid::smem(n, 4096);   // a longer list is sorted in chunks
    }
    return s;
}

}  // namespace

// Float sets: up to 4096 points.  The grid's error (a few 2^-30 of the axes)
// keeps every slope alive whose width is within about 1e-5 of the optimum:
// tens of slopes up to here (0.42 - 0.86 ms against 1.24 at n = 2048, 0.75
// against 2.48 at 4096), thousands above (n = 8192: 1.7 - 9.7 ms against
// 9.2 - 10.3), each scored by a sort.
bool direct_f32_ok(int n, int h) { return n >= 16 && n <= 4096 && (long long)h * 4 >= n; }

// A small order statistic leaves many intervals alive.  Against the paths of
// many kernels, ordinary sets (lines, random points, curves; median and largest
// ratio of times): h = n / 3: batches of 4096-point sets 0.28 and 0.54, single
// fits at 2048 points 0.58 and 1.04; h = n / 4: 0.35 and 15, 0.63 and 1.03;
// h = n / 8: 0.38 and 25, 0.62 and 1.64.
bool direct_ok(int n, int h) { return n >= 2 && n <= 65536 && (long long)h * 3 >= n; }

size_t direct_bytes(int n) { return (size_t)d_up(team_bytes(single_of(n).shape)); }

cudaError_t launch_direct(const short *x, const short *y, int n, int h, int algo, const float *pred, lms_result *out,
                          void *mem, cudaStream_t st)
{
    const Single s = single_of(n);
    DirectArgs a = {};
    a.x = x;
    a.y = y;
    a.n = n;
    a.h = h;
    a.nsets = 1;
    a.algo = algo;
    a.plain_max = 0;
    a.bnb_min = 0x7fffffff;
    a.pred = pred;
    a.out = out;
    a.mem = static_cast<unsigned char *>(mem);
    a.shape = s.shape;
    if (s.variant == 0) return launch_cluster<Small>(a, s.smem, st);
    if (s.variant == 1) return launch_cluster<Mid>(a, s.smem, st);
    return launch_cluster<Large>(a, s.smem, st);
}

// ---------------------------------------------------------------- float sets
size_t direct_f32_bytes(int n) { return (size_t)d_up(team_bytes(float_single_of(n).shape)); }

cudaError_t launch_direct_f32(const float *x, const float *y, int n, int h, int algo, lms_result *out, int *done,
                              void *mem, cudaStream_t st)
{
    const Single s = float_single_of(n);
    DirectArgs a = {};
    a.xf = x;
    a.yf = y;
    a.n = n;
    a.h = h;
    a.nsets = 1;
    a.algo = algo;
    a.bnb_min = 0x7fffffff;
    a.out = out;
    a.done = done;
    a.mem = static_cast<unsigned char *>(mem);
    a.shape = s.shape;
    cudaError_t e = cudaMemsetAsync(done, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    return s.variant == 0 ? launch_cluster<FloatSmall>(a, s.smem, st) : launch_cluster<FloatMid>(a, s.smem, st);
}

// ---------------------------------------------------------------- many sets
namespace {
TeamShape batch_shape(int nmax) { return Batch::team(nmax, 1, 2048, 256.0f); }
}  // namespace

int direct_batch_teams(int nsets, int nmax, int sms)
{
    return std::min(nsets, batch_teams_per_sm(Batch::smem(nmax, batch_shape(nmax).HC)) * sms);
}

size_t direct_batch_bytes(int nteams, int nmax)
{
    return (size_t)team_bytes(batch_shape(nmax)) * nteams + 256;
}

cudaError_t launch_direct_batch(const short *x, const short *y, const long long *off, const int *hvec, const int *sets,
                                int nsets, int nmax, int nteams, int plain_max, int bnb_min, int *set_done,
                                int small_max, lms_result *out, void *mem, cudaStream_t st)
{
    DirectArgs a = {};
    a.x = x;
    a.y = y;
    a.off = off;
    a.hvec = hvec;
    a.sets = sets;
    a.nsets = nsets;
    a.algo = LMS_ALGO_SWEEP;
    a.plain_max = plain_max;
    a.bnb_min = bnb_min;
    a.set_done = set_done;
    a.small_max = small_max;
    a.out = out;
    a.next = static_cast<int *>(mem);
    a.mem = static_cast<unsigned char *>(mem) + 256;
    a.shape = batch_shape(nmax);
    const size_t smem = Batch::smem(nmax, a.shape.HC);
    cudaError_t e = cudaMemsetAsync(a.next, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    return launch_batch(a, nteams, smem, st);
}

}  // namespace lms
