// cnn_api.cpp -- C ABI of the refinement-flag predictor's kernels (forward,
// loss gradient, training) on host buffers.  The network and its use inside
// regridding are described in include/tsunami.h.
#include <cmath>
#include <cstring>
#include <algorithm>
#include <mutex>
#include <random>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/tsunami.h"
#include "cnn.h"

using namespace tsu;

namespace {

// The device buffers of one call, cut out of one allocation from a memory pool of
// the process: cudaMalloc and cudaFree take tens of microseconds each and wait for
// the device, and the calls used up to twelve of both.  The pool (one per device,
// stream-ordered, safe from several threads) keeps at most kPoolKeep bytes between
// calls; what is above that goes back to the device at the next synchronisation, so a
// call that needs more maps the rest anew each time.
constexpr unsigned long long kPoolKeep = 64ull << 20;
constexpr int kMaxDevices = 64;

cudaError_t pool_of_device(cudaMemPool_t *out)
{
    static std::mutex mu;
    static cudaMemPool_t pools[kMaxDevices] = {nullptr};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (!pools[dev]) {
        cudaMemPoolProps p{};
        p.allocType = cudaMemAllocationTypePinned;
        p.location.type = cudaMemLocationTypeDevice;
        p.location.id = dev;
        cudaMemPool_t q = nullptr;
        e = cudaMemPoolCreate(&q, &p);
        if (e != cudaSuccess) return e;
        unsigned long long keep = kPoolKeep;
        e = cudaMemPoolSetAttribute(q, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e != cudaSuccess) {
            cudaMemPoolDestroy(q);
            return e;
        }
        pools[dev] = q;
    }
    *out = pools[dev];
    return cudaSuccess;
}

struct Bufs {
    char *p = nullptr;
    size_t used = 0;
    ~Bufs() { if (p) cudaFreeAsync(p, 0); }
    size_t want(size_t bytes)   // offset of a buffer; all are asked for before alloc()
    {
        const size_t o = used;
        used += (bytes + 255) & ~(size_t)255;
        return o;
    }
    cudaError_t alloc()
    {
        cudaMemPool_t pool = nullptr;
        const cudaError_t e = pool_of_device(&pool);
        if (e != cudaSuccess) return e;
        return cudaMallocFromPoolAsync((void **)&p, used < 256 ? 256 : used, pool, 0);
    }
    template <typename T> T *at(size_t off) const { return reinterpret_cast<T *>(p + off); }
};

#define CKR(x) do { if ((x) != cudaSuccess) return TSU_ERR_CUDA; } while (0)

}  // namespace

extern "C" int tsu_cnn_num_params(void) { return cnn_n_params(); }

extern "C" int tsu_cnn_forward(const float *theta, const float *x, int n, int h, int w, int fp16, float *logits)
{
    if (!theta || !x || !logits || n < 1 || h < 1 || w < 1) return TSU_ERR_ARG;
    const size_t px = (size_t)n * h * w;
    const int np = cnn_n_params();
    Bufs b;
    const size_t oth = b.want(np * sizeof(float)), ox = b.want(px * kCnnIn * sizeof(float)), olog = b.want(px * sizeof(float));
    const size_t oact = b.want(fp16 ? 0 : px * 3 * kCnnHidden * sizeof(float));   // FP32 only
    const size_t ohalf = b.want(fp16 ? cnn_half_workspace_bytes(n, h, w) : 0);
    CKR(b.alloc());
    CKR(cudaMemcpy(b.at<float>(oth), theta, np * sizeof(float), cudaMemcpyHostToDevice));
    CKR(cudaMemcpy(b.at<float>(ox), x, px * kCnnIn * sizeof(float), cudaMemcpyHostToDevice));
    if (cnn_forward(b.at<float>(oth), b.at<float>(ox), n, h, w, fp16 != 0, b.at<float>(oact), b.at<float>(olog),
                    b.at<char>(ohalf), 0))
        return TSU_ERR_CUDA;
    CKR(cudaMemcpy(logits, b.at<float>(olog), px * sizeof(float), cudaMemcpyDeviceToHost));
    return TSU_OK;
}

extern "C" int tsu_cnn_loss_grad(const float *theta, const float *x, const float *t, const float *m, int n, int h,
                                 int w, double *loss, float *grad)
{
    if (!theta || !x || !t || !m || !loss || !grad || n < 1 || h < 1 || w < 1) return TSU_ERR_ARG;
    const size_t px = (size_t)n * h * w;
    const int np = cnn_n_params();
    double cnt = 0.0;
    for (size_t k = 0; k < px; k++) cnt += m[k];
    Bufs b;
    const size_t oth = b.want(np * sizeof(float)), ox = b.want(px * kCnnIn * sizeof(float)), ot = b.want(px * sizeof(float)),
                 om = b.want(px * sizeof(float)), ows = b.want(cnn_workspace_floats(n, h, w) * sizeof(float)),
                 og = b.want(np * sizeof(float)), ol = b.want(sizeof(double));
    CKR(b.alloc());
    CKR(cudaMemcpy(b.at<float>(oth), theta, np * sizeof(float), cudaMemcpyHostToDevice));
    CKR(cudaMemcpy(b.at<float>(ox), x, px * kCnnIn * sizeof(float), cudaMemcpyHostToDevice));
    CKR(cudaMemcpy(b.at<float>(ot), t, px * sizeof(float), cudaMemcpyHostToDevice));
    CKR(cudaMemcpy(b.at<float>(om), m, px * sizeof(float), cudaMemcpyHostToDevice));
    if (cnn_loss_grad(b.at<float>(oth), b.at<float>(ox), b.at<float>(ot), b.at<float>(om), n, h, w, (float)cnt,
                      b.at<float>(ows), b.at<float>(og), b.at<double>(ol), 0))
        return TSU_ERR_CUDA;
    CKR(cudaMemcpy(grad, b.at<float>(og), np * sizeof(float), cudaMemcpyDeviceToHost));
    CKR(cudaMemcpy(loss, b.at<double>(ol), sizeof(double), cudaMemcpyDeviceToHost));
    return TSU_OK;
}

// Mini-batch Adam on the GPU over a host dataset of n planes; batches of
// `batch` planes drawn with a Mersenne twister seeded by `seed`.
extern "C" int tsu_cnn_train(float *theta, const float *x, const float *t, const float *m, int n, int h, int w,
                             int steps, int batch, float lr, unsigned seed, double *loss_first, double *loss_last)
{
    if (!theta || !x || !t || !m || n < 1 || h < 1 || w < 1 || steps < 1 || batch < 1 || !(lr > 0)) return TSU_ERR_ARG;
    if (batch > n) batch = n;
    const size_t plane = (size_t)h * w;
    const int np = cnn_n_params();
    Bufs b_;
    const size_t fb = sizeof(float), np_ = (size_t)n * plane, bp = (size_t)batch * plane;
    const size_t oth = b_.want(np * fb), ox = b_.want(np_ * kCnnIn * fb), ot = b_.want(np_ * fb), om = b_.want(np_ * fb),
                 ows = b_.want(cnn_workspace_floats(batch, h, w) * fb), og = b_.want(np * fb), ol = b_.want(sizeof(double)),
                 omo = b_.want(np * fb), ov = b_.want(np * fb), obx = b_.want(bp * kCnnIn * fb), obt = b_.want(bp * fb),
                 obm = b_.want(bp * fb);
    CKR(b_.alloc());
    float *const dth = b_.at<float>(oth), *const dx = b_.at<float>(ox), *const dt = b_.at<float>(ot), *const dm = b_.at<float>(om);
    float *const dg = b_.at<float>(og), *const dmo = b_.at<float>(omo), *const dv = b_.at<float>(ov);
    float *const bx = b_.at<float>(obx), *const bt = b_.at<float>(obt), *const bm = b_.at<float>(obm);
    double *const dl = b_.at<double>(ol);
    CKR(cudaMemcpy(dth, theta, np * sizeof(float), cudaMemcpyHostToDevice));
    CKR(cudaMemcpy(dx, x, (size_t)n * plane * kCnnIn * sizeof(float), cudaMemcpyHostToDevice));
    CKR(cudaMemcpy(dt, t, (size_t)n * plane * sizeof(float), cudaMemcpyHostToDevice));
    CKR(cudaMemcpy(dm, m, (size_t)n * plane * sizeof(float), cudaMemcpyHostToDevice));
    CKR(cudaMemset(dmo, 0, np * sizeof(float)));
    CKR(cudaMemset(dv, 0, np * sizeof(float)));
    std::vector<double> cnt(n, 0.0);
    for (int k = 0; k < n; k++)
        for (size_t q = 0; q < plane; q++) cnt[k] += m[(size_t)k * plane + q];
    std::mt19937 rng(seed);
    std::vector<int> order(n);
    for (int k = 0; k < n; k++) order[k] = k;
    size_t pos = n;
    for (int s = 1; s <= steps; s++) {
        double bc = 0.0;
        for (int b = 0; b < batch; b++) {
            if (pos >= (size_t)n) { std::shuffle(order.begin(), order.end(), rng); pos = 0; }
            int k = order[pos++];
            bc += cnt[k];
            CKR(cudaMemcpyAsync(bx + (size_t)b * plane * kCnnIn, dx + (size_t)k * plane * kCnnIn,
                                plane * kCnnIn * sizeof(float), cudaMemcpyDeviceToDevice, 0));
            CKR(cudaMemcpyAsync(bt + (size_t)b * plane, dt + (size_t)k * plane,
                                plane * sizeof(float), cudaMemcpyDeviceToDevice, 0));
            CKR(cudaMemcpyAsync(bm + (size_t)b * plane, dm + (size_t)k * plane,
                                plane * sizeof(float), cudaMemcpyDeviceToDevice, 0));
        }
        if (cnn_loss_grad(dth, bx, bt, bm, batch, h, w, (float)bc,
                          b_.at<float>(ows), dg, dl, 0))
            return TSU_ERR_CUDA;
        if (s == 1 && loss_first) CKR(cudaMemcpy(loss_first, dl, sizeof(double), cudaMemcpyDeviceToHost));
        if (cnn_adam(dth, dg, dmo, dv, np, lr, s, 0)) return TSU_ERR_CUDA;
        if (s == steps && loss_last) CKR(cudaMemcpy(loss_last, dl, sizeof(double), cudaMemcpyDeviceToHost));
    }
    CKR(cudaMemcpy(theta, dth, np * sizeof(float), cudaMemcpyDeviceToHost));
    return TSU_OK;
}
