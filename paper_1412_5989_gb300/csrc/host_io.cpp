// cih_ham_build_host: the two-body tables from host memory in, the half-stored
// matrix (Sec. 2, stored in compressed rows as in Sec. 4.1) out to host
// memory, with the copies inside the call and the device-to-host copy of each
// row chunk overlapped with the fill of the next one.
#include <algorithm>
#include <vector>

#include "cih_internal.h"

namespace cih {

int build_host(cih_basis &b, int K, double hw, const float *tbme_h, const double *esp_h, int64_t *rowptr_h,
               int32_t *col_h, float *val_h, int64_t capacity, int64_t *nnz_out, cudaStream_t st)
{
    const int64_t dim = b.dim, tl = b.layout.total;
    const int n_orb = b.s[0].n_orb + b.s[1].n_orb;
    Timer tm("build_host");
    std::vector<void *> bufs;
    auto alloc = [&](void **p, size_t bytes) -> bool {
        // the library pool keeps the blocks mapped for the next call
        if (cudaMallocFromPoolAsync(p, std::max<size_t>(bytes, 16), b.pool, st) != cudaSuccess) {
            (void)cudaGetLastError();
            return false;
        }
        bufs.push_back(*p);
        return true;
    };
    // ends of the row chunks in 64ths of the nonzeros
    constexpr int kChunks = 8;
    static const int kChunkEnd[kChunks] = {1, 4, 10, 20, 31, 42, 53, 64};
    cudaStream_t cs = nullptr;
    cudaEvent_t counted = nullptr;
    std::vector<cudaEvent_t> evs;
    int rc = CIH_OK;
    float *tbme_d = nullptr;
    double *esp_d = nullptr;
    int64_t *rowptr_d = nullptr;
    int32_t *col_d = nullptr;
    float *val_d = nullptr, *work = nullptr;
    int64_t nnz = 0;
    cudaError_t e;
    if (!alloc((void **)&tbme_d, sizeof(float) * (size_t)K * tl) || !alloc((void **)&rowptr_d, sizeof(int64_t) * (dim + 1)) ||
        (esp_h && !alloc((void **)&esp_d, sizeof(double) * n_orb))) {
        rc = fail(CIH_ERR_NOMEM, "build_host: device tables");
        goto done;
    }
    if (tl > 0) cudaMemcpyAsync(tbme_d, tbme_h, sizeof(float) * (size_t)K * tl, cudaMemcpyHostToDevice, st);
    if (esp_h) cudaMemcpyAsync(esp_d, esp_h, sizeof(double) * n_orb, cudaMemcpyHostToDevice, st);
    if ((rc = launch_count(b, rowptr_d, st)) || (rc = launch_scan(b, rowptr_d, st))) goto done;
    e = cudaMemcpyAsync(rowptr_h, rowptr_d, sizeof(int64_t) * (dim + 1), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&counted, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(counted, st);
    if (e != cudaSuccess) { rc = cuda_fail(e, "build_host: row pointers"); goto done; }
    // what does not need the count runs while it does: the working copy of the
    // tables (prepared once for all chunks), the copy stream and its events.  From five
    // sets on a copy is two passes, and the link is slower than the row kernel (us,
    // with / without a copy: 3+4 Nmax=4, one set 522 / 558, four 1,114 / 1,137, seven 1,780 /
    // 1,748; 4+4 Nmax=4 1,420 / 1,430, 3,343 / 3,352, 5,353 / 5,306)
    if (K <= 4 && fill_work_floats(b, K) > 0 && alloc((void **)&work, sizeof(float) * fill_work_floats(b, K)) &&
        (rc = fill_prepare(b, K, hw, tbme_d, esp_d, nullptr, work, st)))
        goto done;
    e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) { cs = nullptr; rc = cuda_fail(e, "build_host: copy stream"); goto done; }
    for (int c = 0; c < kChunks; ++c) {
        cudaEvent_t ev;
        if ((e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) != cudaSuccess) {
            rc = cuda_fail(e, "build_host: event");
            goto done;
        }
        evs.push_back(ev);
    }
    e = cudaEventSynchronize(counted);
    if (e != cudaSuccess) { rc = cuda_fail(e, "build_host: row pointers"); goto done; }
    nnz = rowptr_h[dim];
    if (nnz_out) *nnz_out = nnz;
    tm.mark("tables in, count, row pointers out");
    if (nnz > capacity) {
        rc = fail(CIH_ERR_CAPACITY, "build_host: " + std::to_string(nnz) + " stored nonzeros, capacity " +
                                        std::to_string(capacity));
        goto done;
    }
    // the matrix comes before the working copy where the device has no room for both
    while (!((col_d || alloc((void **)&col_d, sizeof(int32_t) * (size_t)nnz)) &&
             alloc((void **)&val_d, sizeof(float) * (size_t)K * nnz)) && work) {
        bufs.erase(std::find(bufs.begin(), bufs.end(), (void *)work));
        cudaFreeAsync(work, st);
        work = nullptr;
    }
    if (!val_d) {
        rc = fail(CIH_ERR_NOMEM, "build_host: device matrix");
        goto done;
    }
    tm.mark_sync("device matrix allocated", st);
    {
        // row chunks; chunk c's copies wait for its fill.  The fill is four to five
        // times faster than the link, so the first chunks are small (the copies
        // start early) and each is filled while the one before it is copied.
        const int C = (int)std::max<int64_t>(1, std::min<int64_t>(kChunks, dim));
        std::vector<int64_t> rb(C + 1, dim);
        rb[0] = 0;
        for (int c = 1; c < C; ++c)
            rb[c] = std::lower_bound(rowptr_h, rowptr_h + dim + 1, nnz * kChunkEnd[c - 1] / 64) - rowptr_h;
        for (int c = 0; c < C && !rc; ++c) {
            const int64_t r0 = std::min(rb[c], dim), r1 = c == C - 1 ? dim : std::max(r0, std::min(rb[c + 1], dim));
            if ((rc = launch_fill(b, rowptr_d, K, hw, tbme_d, false, false, esp_d, col_d, val_d, st, r0, r1, false, nullptr, work, false)))
                break;
            const cudaEvent_t ev = evs[c];
            cudaEventRecord(ev, st);
            cudaStreamWaitEvent(cs, ev, 0);
            const int64_t e0 = rowptr_h[r0], e1 = rowptr_h[r1];
            if (e1 > e0) {
                cudaMemcpyAsync(col_h + e0, col_d + e0, sizeof(int32_t) * (e1 - e0), cudaMemcpyDeviceToHost, cs);
                for (int k = 0; k < K; ++k)
                    cudaMemcpyAsync(val_h + (int64_t)k * capacity + e0, val_d + (int64_t)k * nnz + e0,
                                    sizeof(float) * (e1 - e0), cudaMemcpyDeviceToHost, cs);
            }
        }
        tm.mark_sync("fill chunks done", st);
        e = cudaStreamSynchronize(cs);
        tm.mark("copies done");
        if (!rc && e != cudaSuccess) rc = cuda_fail(e, "build_host: copies");
        e = cudaGetLastError();
        if (!rc && e != cudaSuccess) rc = cuda_fail(e, "build_host");
    }
done:
    for (void *p : bufs) cudaFreeAsync(p, st);
    e = cudaStreamSynchronize(st);
    if (!rc && e != cudaSuccess) rc = cuda_fail(e, "build_host");
    for (cudaEvent_t ev : evs) cudaEventDestroy(ev);
    if (counted) cudaEventDestroy(counted);
    if (cs) cudaStreamDestroy(cs);
    return rc;
}

}  // namespace cih
