// C ABI of the super-potential solver: plan creation and validation, precompute
// (Alg. 1), solves (Alg. 2), diagnostics.  See include/superpot.h for the contract.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <new>
#include <vector>

#include "sp_internal.h"

static thread_local char g_err[1024] = "";

void sp_clear_error(void) { g_err[0] = 0; }

sp_status sp_fail(sp_status st, const char* fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return st;
}

sp_status sp_cuda_check(cudaError_t e, const char* what)
{
    if (e == cudaSuccess) return SP_OK;
    return sp_fail(e == cudaErrorMemoryAllocation ? SP_ERR_OOM : SP_ERR_CUDA, "%s: %s (%s)", what,
                   cudaGetErrorName(e), cudaGetErrorString(e));
}

sp_status sp_plan_alloc(sp_plan p, void** ptr, size_t bytes, const char* what)
{
    *ptr = nullptr;
    if (p->nalloc >= (int)(sizeof(p->alloc_ptr) / sizeof(p->alloc_ptr[0])))
        return sp_fail(SP_ERR_INVALID, "internal: too many plan allocations (%s)", what);
    void* q = nullptr;
    if (p->has_alloc) {
        q = p->alloc.alloc(bytes, p->device, p->alloc.ctx);
        if (!q) return sp_fail(SP_ERR_OOM, "allocator returned NULL for %s (%zu bytes)", what, bytes);
    } else {
        // stream-ordered on the plan's private stream, complete before the pointer is used
        cudaError_t e = cudaMallocAsync(&q, bytes, p->mem_st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(p->mem_st);
        if (e != cudaSuccess) {
            cudaGetLastError();  // allocation failures are not sticky: clear them
            return sp_fail(e == cudaErrorMemoryAllocation ? SP_ERR_OOM : SP_ERR_CUDA,
                           "cudaMallocAsync %s (%zu bytes): %s", what, bytes, cudaGetErrorName(e));
        }
    }
    p->alloc_ptr[p->nalloc] = q;
    p->alloc_bytes[p->nalloc] = bytes;
    ++p->nalloc;
    *ptr = q;
    return SP_OK;
}

// Release everything the plan owns, with the plan's device current.  Device memory of the
// library's own allocations is freed stream-ordered after the plan's last recorded work
// (no host wait); a caller's allocator gets its blocks back only after that work has
// completed (a host wait on the plan's event, not on the device).  Returns the status of
// that wait.
static cudaError_t free_plan(sp_plan p)
{
    if (!p) return cudaSuccess;
    cudaError_t err = cudaSuccess;
    if (p->has_alloc) {
        if (p->done_recorded) err = cudaEventSynchronize(p->done);
        for (int i = p->nalloc - 1; i >= 0; --i)
            p->alloc.release(p->alloc_ptr[i], p->alloc_bytes[i], p->device, p->alloc.ctx);
    } else if (p->mem_st) {
        if (p->done_recorded) err = cudaStreamWaitEvent(p->mem_st, p->done, 0);
        for (int i = p->nalloc - 1; i >= 0; --i) cudaFreeAsync(p->alloc_ptr[i], p->mem_st);
        cudaStreamDestroy(p->mem_st);  // released once its frees have run
    }
    if (p->ev) {
        for (cudaEvent_t e : *p->ev) cudaEventDestroy(e);
        delete p->ev;
    }
    if (p->done) cudaEventDestroy(p->done);
    if (p->staged) {
        for (int i = 0; i < 2; ++i)
            if (p->copy_st[i]) cudaStreamDestroy(p->copy_st[i]);
        for (int i = 0; i < 6; ++i)
            if (p->stage_ev[i]) cudaEventDestroy(p->stage_ev[i]);
    }
    free(p->h_gs_a);
    delete p;
    return err;
}

static const int kMaxLen = 2048;  // largest padded FFT length 2n per axis
static const int kGsCap = 4096;   // largest generated GS table

extern "C" sp_status sp_plan_create(sp_plan* out, const int n[3], const double box_lo[3],
                                    const double box_hi[3], int padding, const double* gs_w,
                                    const double* gs_a, int gs_terms, double eps,
                                    sp_precision prec, int max_batch)
{
    return sp_plan_create_ex(out, n, box_lo, box_hi, padding, gs_w, gs_a, gs_terms, eps, prec, max_batch, nullptr);
}

int sp_f_length(int N)
{
#define SP_F_AT_LEAST(L) \
    if (N <= L) return L;
    SP_F_LENGTHS(SP_F_AT_LEAST)
#undef SP_F_AT_LEAST
    return 0;
}

// Time of an FP64 solve of `batch` right-hand sides on lengths F over that on 2n, from a fit to
// 706 measured solves (2 to 1000 points an axis, batches up to 15000; standard deviation 14 % on
// F, 23 % on 2n): launches and latency (us), then the columns that the tiles hold, empty ones
// included, times their length and a cost an element (ps): by stages on 2n, by the transform's
// operations on F.
static double fp64_longer_ratio(const int N[3], const int F[3], int batch)
{
    const auto up = [](long long a, int b) { return (double)((a + b - 1) / b * b); };
    const long long n0 = N[0] / 2, n1 = N[1] / 2, n2 = N[2] / 2;
    double longer = 0.0, own = 0.0;
    for (int ax = 0; ax < 3; ++ax) {
        RadixPlan rp;
        const bool blue = !sp_radix_plan(N[ax], &rp);
        int rows = N[ax];
        if (blue) {
            for (rows = 1; rows < 2 * N[ax] - 1;) rows *= 2;
            sp_radix_plan(rows, &rp);
        }
        const int tile = sp_line_tile(rows, sizeof(cpx<double>)), tileF = F[ax] <= 48 ? 16 : (F[ax] < 216 ? 8 : 4);
        const long long outer = ax == 1 ? n0 : N[1], outerF = ax == 1 ? n0 : F[1];
        const double lines = ax == 2 ? 2 * up((n0 * n1 + 1) / 2, tile) : 2 * outer * up(n2 + 1, tile);
        const double linesF = ax == 2 ? (double)(n0 * n1) : 2 * outerF * up(F[2] / 2 + 1, tileF);
        own += lines * (rows * (1.8 + 17.3 * rp.nst) * (blue ? 2.56 : 1.0) + (ax == 2 ? 183.0 * N[2] : 0.0));
        longer += linesF * F[ax] * 5.23 * log2((double)F[ax]);
    }
    return (34.0 + 1e-6 * batch * longer) / (90.0 + 1e-6 * batch * own);
}

// A grid takes the lengths F unless every padded length has its tuned plan, or the padding to
// F costs more than the register engine gains over the runtime-radix passes: flat grids, whose
// short axes round up by up to 8 times, and a few cubes (2 to 5, 9 and 10 points an axis in every
// type; 49, 50, 525, 784, 800, 810 and 840 in FP64, where F^3 is up to 2.2 times (2n)^3).  Gains
// at equal work: about 2 in FP64 (pipe-bound in both), 2.5 in double-float, 4 and more in FP32,
// four times that where an axis needs Bluestein's algorithm (512x512x3, growth 2.7: FP64 0.53,
// double-float 0.96, FP32 1.73 times the speed; 129^3: 11, 12 and 18 times).  Grids of up to
// 32^3 points are bound by latency and gain at any growth measured (7x9x5, growth 3.3: 1.3-1.6).
// In FP64, bound by its pipe in both engines, what the padding adds is paid in full once a batch
// fills the chip, and by grids with one Bluestein axis that holds little of the work: there the
// measured times decide.  Of 706 solves 32 had become slower (100x2x11, batch 909, 3.81 -> 8.67
// ms; 20x4x10, batch 2500, 2.45 -> 4.58; 784x2x436 1.43 -> 2.53); at a predicted 0.83 none does,
// and 34 give up gains of up to 41 %, 19 % in the median.  In double-float and FP32 none of 1423
// solves was slower on F.
bool sp_embeds(const int N[3], sp_precision prec, int max_batch, int F[3])
{
    bool tuned = true, blue = false;
    double growth = 1.0;
    for (int ax = 0; ax < 3; ++ax) {
        const bool own = sp_v2_supported(N[ax]);
        F[ax] = own ? N[ax] : sp_f_length(N[ax]);
        if (!F[ax]) return false;
        RadixPlan rp;
        tuned = tuned && own;
        blue = blue || !sp_radix_plan(N[ax], &rp);
        growth *= (double)F[ax] / N[ax];
    }
    const bool small = (long long)N[0] * N[1] * N[2] <= 8LL * 32 * 32 * 32;
    double limit = prec == SP_FP64 ? 1.8 : (prec == SP_DF32 ? 2.5 : 4.0);
    if (blue) limit *= 4.0;
    else if (small) limit = 4.0;
    return !tuned && growth <= limit && (prec != SP_FP64 || fp64_longer_ratio(N, F, max_batch) <= 0.83);
}

static sp_status create_plan(sp_plan* out, const int n[3], const double box_lo[3],
                             const double box_hi[3], int padding, const double* gs_w,
                             const double* gs_a, int gs_terms, double eps,
                             sp_precision prec, int max_batch, const sp_allocator* allocator, bool may_embed);

extern "C" sp_status sp_plan_create_ex(sp_plan* out, const int n[3], const double box_lo[3],
                                       const double box_hi[3], int padding, const double* gs_w,
                                       const double* gs_a, int gs_terms, double eps,
                                       sp_precision prec, int max_batch, const sp_allocator* allocator)
{
    const sp_status rc = create_plan(out, n, box_lo, box_hi, padding, gs_w, gs_a, gs_terms, eps, prec, max_batch,
                                     allocator, true);
    // the longer transforms need a larger workspace: without the memory, the 2n passes
    if (rc != SP_ERR_OOM) return rc;
    int N[3], F[3];
    for (int ax = 0; ax < 3; ++ax) N[ax] = 2 * n[ax];
    if (!sp_embeds(N, prec, max_batch, F)) return rc;
    return create_plan(out, n, box_lo, box_hi, padding, gs_w, gs_a, gs_terms, eps, prec, max_batch, allocator, false);
}

sp_status sp_plan_create_2n(sp_plan* out, const int n[3], const double box_lo[3], const double box_hi[3], double eps,
                            sp_precision prec, int max_batch)
{
    return create_plan(out, n, box_lo, box_hi, 2, nullptr, nullptr, 0, eps, prec, max_batch, nullptr, false);
}

// What the sizes of a plan's buffers depend on: lengths, strides and the GS table's length
// (0 gs_terms: generated).  Host only.
static void plan_geometry(sp_plan p, const int n[3], const double box_lo[3], const double box_hi[3], int gs_terms,
                          double eps, sp_precision prec, int max_batch, bool may_embed)
{
    for (int ax = 0; ax < 3; ++ax) {
        p->n[ax] = n[ax];
        p->N[ax] = 2 * n[ax];
        p->lo[ax] = box_lo[ax];
        p->hi[ax] = box_hi[ax];
        p->h[ax] = (box_hi[ax] - box_lo[ax]) / (n[ax] - 1);
        p->L[ax] = n[ax] * p->h[ax];
        // a padded length with a prime factor above 7 has no radix plan: Bluestein's
        // algorithm, a circular convolution of length M = 2^k >= 2N - 1
        if (!sp_radix_plan(p->N[ax], &p->rp[ax])) {
            p->rp[ax].nst = 0;
            int M = 1;
            while (M < 2 * p->N[ax] - 1) M *= 2;
            p->blue_M[ax] = M;
            sp_radix_plan(M, &p->blue_rp[ax]);
        }
    }
    p->prec = prec;
    p->max_batch = max_batch;
    p->ldz = (n[2] + 1 + 7) & ~7;
    p->plane = 2LL * n[1] * p->ldz;
    const size_t csize = (prec == SP_FP64 || prec == SP_DF32) ? 16 : 8;
    p->emb = sp_embeds(p->N, prec, max_batch, p->F) && may_embed;
    if (!p->emb)
        for (int ax = 0; ax < 3; ++ax) p->F[ax] = p->N[ax];
    p->ldf = (p->F[2] / 2 + 1 + 7) & ~7;
    p->planef = (long long)p->F[1] * p->ldf;
    p->keep_n = p->emb && csize * n[0] * p->plane <= SP_NOALLOC_MAX_BYTES && csize * n[0] * p->planef > SP_NOALLOC_MAX_BYTES;
    p->work_bytes = csize * (size_t)max_batch * n[0] * (size_t)p->planef;
    p->eps = eps;
    p->delta = sqrt(p->L[0] * p->L[0] + p->L[1] * p->L[1] + p->L[2] * p->L[2]);
    p->h_tau = 0.1;
    p->eta = 1e-17;
    p->gs_user = gs_terms > 0;
    // the generated table's length is fixed by eps and delta (eq. sin_1_x): known now
    p->gs_cap = p->gs_terms = p->gs_user ? gs_terms : sp_gs_terms(p);
}

// Every device buffer that a plan holds, in the order of allocation: visit(pointer, bytes,
// name) for each, up to the first failure.  The one list behind creation and sp_plan_bytes.
template <class Visit> static sp_status plan_buffers(sp_plan p, Visit&& visit)
{
    sp_status rc;
#define SP_BUFFER(ptr, bytes) \
    if ((rc = visit((void**)&(ptr), (size_t)(bytes), #ptr))) return rc
    const size_t csize = (p->prec == SP_FP64 || p->prec == SP_DF32) ? 16 : 8;
    SP_BUFFER(p->d_status, 256);
    SP_BUFFER(p->d_gs_w, sizeof(double) * p->gs_cap);
    SP_BUFFER(p->d_gs_a, sizeof(double) * p->gs_cap);
    // 1D integral tables [s][k] per axis; axes with the same (n, L) share one
    for (int ax = 0; ax < 3; ++ax) {
        int same = -1;
        for (int q = 0; q < ax; ++q)
            if (p->n[q] == p->n[ax] && p->L[q] == p->L[ax]) { same = q; break; }
        if (same >= 0) {
            p->d_G[ax] = p->d_G[same];
            p->d_H[ax] = p->d_H[same];
            continue;
        }
        const size_t tb = sizeof(double) * (size_t)p->gs_cap * (p->n[ax] + 1);
        SP_BUFFER(p->d_G[ax], tb);
        SP_BUFFER(p->d_H[ax], tb);
    }
    const size_t mcount = (size_t)(p->n[0] + 1) * (p->n[1] + 1) * p->ldz;
    SP_BUFFER(p->d_M64, sizeof(double) * mcount);
    if (!p->emb || p->keep_n) {
        if (p->prec == SP_FP32 || p->prec == SP_MIXED) SP_BUFFER(p->d_M32, sizeof(float) * mcount);
        if (p->prec == SP_DF32) SP_BUFFER(p->d_Mdf, sizeof(df32) * mcount);
    }
    if (p->emb) {
        SP_BUFFER(p->d_Ms, csize / 2 * (size_t)(p->F[0] / 2 + 1) * (p->F[1] / 2 + 1) * p->ldf);
        for (int ax = 0; ax < 3; ++ax)
            if (!sp_v2_supported(p->N[ax])) SP_BUFFER(p->d_twF[ax], csize * (p->F[ax] + SP_TW_STAGED_MAX));
    }
    for (int ax = 0; ax < 3; ++ax) {
        SP_BUFFER(p->d_tw64[ax], sizeof(cpx<double>) * p->N[ax]);
        SP_BUFFER(p->d_tw32[ax], sizeof(cpx<float>) * (p->N[ax] + SP_TW_STAGED_MAX));
        SP_BUFFER(p->d_twdf[ax], sizeof(cpx<df32>) * (p->N[ax] + SP_TW_STAGED_MAX));
    }
    for (int ax = 0; ax < 3; ++ax)
        if (p->blue_M[ax]) SP_BUFFER(p->d_blue[ax], sp_bluestein_bytes(p, ax));
    SP_BUFFER(p->d_work, p->work_bytes);
#undef SP_BUFFER
    return SP_OK;
}

size_t sp_plan_bytes(const int n[3], const double box_lo[3], const double box_hi[3], double eps, sp_precision prec,
                     int max_batch, bool may_embed)
{
    sp_plan_s view = {};
    plan_geometry(&view, n, box_lo, box_hi, 0, eps, prec, max_batch, may_embed);
    if (view.gs_cap < 1 || view.gs_cap > kGsCap) view.gs_cap = 0;  // creation refuses the plan
    size_t total = 0;
    plan_buffers(&view, [&](void**, size_t bytes, const char*) {
        total += bytes;
        return SP_OK;
    });
    return total;
}

static sp_status create_plan(sp_plan* out, const int n[3], const double box_lo[3],
                             const double box_hi[3], int padding, const double* gs_w,
                             const double* gs_a, int gs_terms, double eps,
                             sp_precision prec, int max_batch, const sp_allocator* allocator, bool may_embed)
{
    g_err[0] = 0;
    if (!out) return sp_fail(SP_ERR_INVALID, "out is NULL");
    *out = nullptr;
    if (!n || !box_lo || !box_hi) return sp_fail(SP_ERR_INVALID, "n, box_lo and box_hi must be non-NULL");
    if (padding != 2) return sp_fail(SP_ERR_INVALID, "padding must be 2 (got %d)", padding);
    if (prec != SP_FP64 && prec != SP_FP32 && prec != SP_MIXED && prec != SP_DF32)
        return sp_fail(SP_ERR_INVALID, "unknown precision %d", (int)prec);
    if (max_batch < 1) return sp_fail(SP_ERR_INVALID, "max_batch must be >= 1 (got %d)", max_batch);
    if (allocator && (!allocator->alloc || !allocator->release))
        return sp_fail(SP_ERR_INVALID, "allocator: both alloc and release must be given");
    for (int ax = 0; ax < 3; ++ax) {
        if (n[ax] < 2 || 2 * n[ax] > kMaxLen)
            return sp_fail(SP_ERR_UNSUPPORTED_SIZE, "n[%d] = %d: need n >= 2 and 2n <= %d", ax, n[ax], kMaxLen);
        if (!(isfinite(box_lo[ax]) && isfinite(box_hi[ax]) && box_hi[ax] > box_lo[ax]))
            return sp_fail(SP_ERR_INVALID, "box axis %d: need finite lo < hi", ax);
    }
    const bool user = gs_w || gs_a || gs_terms;
    if (user) {
        if (!gs_w || !gs_a || gs_terms < 1)
            return sp_fail(SP_ERR_INVALID, "GS table: give both arrays and gs_terms >= 1, or none");
        for (int s = 0; s < gs_terms; ++s)
            if (!(isfinite(gs_w[s]) && isfinite(gs_a[s]) && gs_a[s] > 0.0))
                return sp_fail(SP_ERR_INVALID, "GS table entry %d is not finite with a > 0", s);
    } else if (!(eps > 0.0 && eps < 1.0)) {
        return sp_fail(SP_ERR_INVALID, "eps must be in (0, 1) (got %g)", eps);
    }

    sp_plan p = new (std::nothrow) sp_plan_s();
    if (!p) return sp_fail(SP_ERR_OOM, "host allocation failed");
    cudaGetDevice(&p->device);
    if (allocator) {
        p->alloc = *allocator;
        p->has_alloc = true;
    }
    plan_geometry(p, n, box_lo, box_hi, user ? gs_terms : 0, eps, prec, max_batch, may_embed);
    const int terms = p->gs_terms;
    if (!user && (terms < 1 || terms > kGsCap)) {
        delete p;
        return sp_fail(SP_ERR_INVALID, "GS table of %d terms (eps %g): at most %d", terms, eps, kGsCap);
    }

    p->ev = new (std::nothrow) std::vector<cudaEvent_t>();
    p->h_gs_a = (double*)malloc(sizeof(double) * p->gs_cap);
    if (!p->h_gs_a || !p->ev) {
        free_plan(p);
        return sp_fail(SP_ERR_OOM, "host allocation failed");
    }
    if (user) memcpy(p->h_gs_a, gs_a, sizeof(double) * gs_terms);
    else sp_gs_exponents(p, p->h_gs_a);
    sp_status rc = SP_OK;
    if ((rc = sp_cuda_check(cudaEventCreateWithFlags(&p->done, cudaEventDisableTiming), "create plan event"))) {
        p->done = nullptr;
        free_plan(p);
        return rc;
    }
    if (!p->has_alloc &&
        (rc = sp_cuda_check(cudaStreamCreateWithFlags(&p->mem_st, cudaStreamNonBlocking), "create plan stream"))) {
        p->mem_st = nullptr;
        free_plan(p);
        return rc;
    }
    if ((rc = plan_buffers(p, [p](void** ptr, size_t bytes, const char* what) { return sp_plan_alloc(p, ptr, bytes, what); }))) {
        free_plan(p);
        return rc;
    }
    for (int ax = 0; ax < 3; ++ax) {  // Bluestein tables: built on the host, copied once
        if (!p->blue_M[ax]) continue;
        std::vector<unsigned char> host(sp_bluestein_bytes(p, ax));
        sp_bluestein_fill(p, ax, host.data());
        // pageable source: the call returns once the bytes are staged, so host may go
        const cudaError_t ce = p->mem_st ? cudaMemcpyAsync(p->d_blue[ax], host.data(), host.size(),
                                                           cudaMemcpyHostToDevice, p->mem_st)
                                         : cudaMemcpy(p->d_blue[ax], host.data(), host.size(), cudaMemcpyHostToDevice);
        if ((rc = sp_cuda_check(ce, "Bluestein tables"))) {
            free_plan(p);
            return rc;
        }
    }
    const cudaError_t ce = p->mem_st ? cudaMemsetAsync(p->d_status, 0, 256, p->mem_st) : cudaMemset(p->d_status, 0, 256);
    if ((rc = sp_cuda_check(ce == cudaSuccess && p->mem_st ? cudaStreamSynchronize(p->mem_st) : ce,
                            "clear status word"))) {
        free_plan(p);
        return rc;
    }
    if (user) {
        if ((rc = sp_cuda_check(cudaMemcpy(p->d_gs_w, gs_w, sizeof(double) * gs_terms, cudaMemcpyHostToDevice),
                                "copy GS weights")) ||
            (rc = sp_cuda_check(cudaMemcpy(p->d_gs_a, gs_a, sizeof(double) * gs_terms, cudaMemcpyHostToDevice),
                                "copy GS exponents"))) {
            free_plan(p);
            return rc;
        }
    }
    *out = p;
    return SP_OK;
}

sp_status sp_record_done(sp_plan p, cudaStream_t st)
{
    sp_status rc = sp_cuda_check(cudaEventRecord(p->done, st), "record plan event");
    if (rc == SP_OK) p->done_recorded = true;
    return rc;
}

extern "C" sp_status sp_kernel_precompute(sp_plan p, sp_stream stream)
{
    g_err[0] = 0;
    if (!p) return sp_fail(SP_ERR_INVALID, "plan is NULL");
    cudaStream_t st = (cudaStream_t)stream;
    sp_status rc = sp_check_device(p);
    if (rc) return rc;
    const size_t mcount = (size_t)(p->n[0] + 1) * (p->n[1] + 1) * p->ldz;
    if ((rc = sp_cuda_check(cudaMemsetAsync(p->d_M64, 0, sizeof(double) * mcount, st), "clear multiplier")))
        return rc;
    if ((rc = sp_setup_run(p, st))) return rc;
    if ((rc = sp_record_done(p, st))) return rc;
    p->ready = true;
    return SP_OK;
}

extern "C" sp_status sp_plan_set_kernel(sp_plan p, sp_kernel kind)
{
    g_err[0] = 0;
    if (!p) return sp_fail(SP_ERR_INVALID, "plan is NULL");
    if (kind != SP_KERNEL_SUPERPOTENTIAL && kind != SP_KERNEL_GS_PLAIN)
        return sp_fail(SP_ERR_INVALID, "unknown kernel %d", (int)kind);
    p->kernel = (int)kind;
    p->ready = false;
    return SP_OK;
}

// The plan's memory lives on the device it was created on; launching its passes while
// another device is current would hand that device foreign pointers.
sp_status sp_check_device(const sp_plan p)
{
    int dev = -1;
    sp_status rc = sp_cuda_check(cudaGetDevice(&dev), "current device");
    if (rc) return rc;
    if (dev != p->device)
        return sp_fail(SP_ERR_INVALID, "plan was created on device %d, current device is %d", p->device, dev);
    return SP_OK;
}

static sp_status check_solve_args(sp_plan p, const void* rho, const void* u)
{
    if (!p) return sp_fail(SP_ERR_INVALID, "plan is NULL");
    if (!rho || !u) return sp_fail(SP_ERR_INVALID, "rho and u must be non-NULL device pointers");
    if (!p->ready) return sp_fail(SP_ERR_NOT_READY, "sp_kernel_precompute has not been run on this plan");
    return sp_check_device(p);
}

extern "C" sp_status sp_solve(sp_plan p, const void* rho, void* u, sp_stream stream)
{
    g_err[0] = 0;
    sp_status rc = check_solve_args(p, rho, u);
    if (rc) return rc;
    if ((rc = sp_run_solve(p, rho, u, 1, (cudaStream_t)stream))) return rc;
    return sp_record_done(p, (cudaStream_t)stream);
}

extern "C" sp_status sp_solve_batched(sp_plan p, const void* rho, void* u, int batch, sp_stream stream)
{
    g_err[0] = 0;
    sp_status rc = check_solve_args(p, rho, u);
    if (rc) return rc;
    if (batch < 1 || batch > p->max_batch)
        return sp_fail(SP_ERR_INVALID, "batch %d outside [1, max_batch = %d]", batch, p->max_batch);
    if ((rc = sp_run_solve(p, rho, u, batch, (cudaStream_t)stream))) return rc;
    return sp_record_done(p, (cudaStream_t)stream);
}

extern "C" sp_status sp_forward_spectrum(sp_plan p, const void* rho, void* spec, sp_stream stream)
{
    g_err[0] = 0;
    sp_status rc = check_solve_args(p, rho, spec);
    if (rc) return rc;
    if ((rc = sp_run_forward(p, rho, spec, (cudaStream_t)stream))) return rc;
    return sp_record_done(p, (cudaStream_t)stream);
}

extern "C" sp_status sp_plan_destroy(sp_plan p)
{
    g_err[0] = 0;
    if (!p) return SP_OK;
    // wait for the plan's own last work and free on the plan's device, whichever device is
    // current
    int cur = -1;
    const bool switched = cudaGetDevice(&cur) == cudaSuccess && cur != p->device &&
                          cudaSetDevice(p->device) == cudaSuccess;
    cudaError_t e = free_plan(p);
    if (switched) cudaSetDevice(cur);
    return sp_cuda_check(e, "order the plan's release after its work");
}

extern "C" sp_status sp_plan_sync(sp_plan p)
{
    g_err[0] = 0;
    if (!p) return sp_fail(SP_ERR_INVALID, "plan is NULL");
    sp_status rc = sp_check_device(p);
    if (rc) return rc;
    if (p->done_recorded && (rc = sp_cuda_check(cudaEventSynchronize(p->done), "wait for the plan's work")))
        return rc;
    if ((rc = sp_cuda_check(cudaGetLastError(), "pending device error"))) return rc;
    int status = 0;
    if ((rc = sp_cuda_check(cudaMemcpy(&status, p->d_status, sizeof(int), cudaMemcpyDeviceToHost), "read status word")))
        return rc;
    if (status != 0) {
        if ((rc = sp_cuda_check(cudaMemset(p->d_status, 0, sizeof(int)), "clear status word"))) return rc;
        return sp_fail(SP_ERR_TIMEOUT, "a bounded device wait gave up (status %d): some work of the solve was not done",
                       status);
    }
    return SP_OK;
}

extern "C" size_t sp_plan_workspace_bytes(const sp_plan p) { return p ? p->work_bytes : 0; }

extern "C" int sp_plan_gs_terms(const sp_plan p) { return p ? p->gs_terms : 0; }

extern "C" sp_status sp_plan_copy_tables(sp_plan p, double* gs_w, double* gs_a, double* M, int axis,
                                         double* G, double* H)
{
    g_err[0] = 0;
    if (!p) return sp_fail(SP_ERR_INVALID, "plan is NULL");
    if (!p->ready) return sp_fail(SP_ERR_NOT_READY, "sp_kernel_precompute has not been run on this plan");
    if ((G || H) && (axis < 0 || axis > 2)) return sp_fail(SP_ERR_INVALID, "axis must be 0, 1 or 2");
    sp_status rc;
    if ((rc = sp_check_device(p))) return rc;
    if (p->done_recorded && (rc = sp_cuda_check(cudaEventSynchronize(p->done), "wait for the plan's work")))
        return rc;
    const int S = p->gs_terms;
    if (gs_w && (rc = sp_cuda_check(cudaMemcpy(gs_w, p->d_gs_w, sizeof(double) * S, cudaMemcpyDeviceToHost),
                                    "copy GS weights")))
        return rc;
    if (gs_a && (rc = sp_cuda_check(cudaMemcpy(gs_a, p->d_gs_a, sizeof(double) * S, cudaMemcpyDeviceToHost),
                                    "copy GS exponents")))
        return rc;
    if (M) {
        const int n0p = p->n[0] + 1, n1p = p->n[1] + 1, n2p = p->n[2] + 1;
        std::vector<double> dev((size_t)n0p * n1p * p->ldz);
        if ((rc = sp_cuda_check(cudaMemcpy(dev.data(), p->d_M64, sizeof(double) * dev.size(),
                                           cudaMemcpyDeviceToHost), "copy multiplier")))
            return rc;
        for (int k0 = 0; k0 < n0p; ++k0)
            for (int k1 = 0; k1 < n1p; ++k1)
                for (int k2 = 0; k2 < n2p; ++k2)
                    M[((size_t)k0 * n1p + k1) * n2p + k2] = dev[((size_t)k1 * n0p + k0) * p->ldz + k2];
    }
    const size_t tb = sizeof(double) * (size_t)S * (p->n[axis < 0 ? 0 : axis] + 1);
    if (G && (rc = sp_cuda_check(cudaMemcpy(G, p->d_G[axis], tb, cudaMemcpyDeviceToHost), "copy G"))) return rc;
    if (H && (rc = sp_cuda_check(cudaMemcpy(H, p->d_H[axis], tb, cudaMemcpyDeviceToHost), "copy H"))) return rc;
    return SP_OK;
}

sp_status sp_mark(sp_plan p, cudaStream_t st)
{
    if (!p->timing) return SP_OK;
    std::vector<cudaEvent_t>& ev = *p->ev;
    if (p->ev_used == ev.size()) {  // the pool is exhausted: grow it (outside a reserved record)
        cudaEvent_t e;
        sp_status rc = sp_cuda_check(cudaEventCreate(&e), "create timing event");
        if (rc) return rc;
        ev.push_back(e);
    }
    return sp_cuda_check(cudaEventRecord(ev[p->ev_used++], st), "record timing event");
}

// Events for `solves` recorded solves (npass + 1 each; 8 passes assumed before the first
// solve tells the pass count).
static sp_status reserve_events(sp_plan p, int solves)
{
    const int per = (p->npass > 0 ? p->npass : 8) + 1;
    const size_t want = p->ev_used + (size_t)solves * per;
    std::vector<cudaEvent_t>& ev = *p->ev;
    while (ev.size() < want) {
        cudaEvent_t e;
        sp_status rc = sp_cuda_check(cudaEventCreate(&e), "create timing event");
        if (rc) return rc;
        ev.push_back(e);
    }
    return SP_OK;
}

extern "C" sp_status sp_plan_set_timing(sp_plan p, int enable)
{
    g_err[0] = 0;
    if (!p) return sp_fail(SP_ERR_INVALID, "plan is NULL");
    if (enable < 0) return sp_fail(SP_ERR_INVALID, "enable must be >= 0 (got %d)", enable);
    p->timing = enable != 0;
    if (enable > 0) return reserve_events(p, enable);
    return SP_OK;
}

extern "C" int sp_plan_pass_times(sp_plan p, double* total_ms, int* launches, const char** names,
                                  int max_passes)
{
    g_err[0] = 0;
    if (!p) { sp_fail(SP_ERR_INVALID, "plan is NULL"); return -1; }
    const int np = p->npass;
    const int per = np + 1;
    for (int i = 0; i < max_passes && i < np; ++i) {
        if (total_ms) total_ms[i] = 0.0;
        if (launches) launches[i] = 0;
        if (names) names[i] = p->pass_name[i];
    }
    std::vector<cudaEvent_t>& ev = *p->ev;
    const size_t used = p->ev_used;
    if (np == 0 || used == 0) return np;
    if (used % per != 0) { sp_fail(SP_ERR_INVALID, "incomplete timing record"); return -1; }
    if (sp_cuda_check(cudaEventSynchronize(ev[used - 1]), "wait for timing events")) return -1;
    for (size_t s0 = 0; s0 < used; s0 += per) {
        for (int i = 0; i < np; ++i) {
            float ms = 0.f;
            if (sp_cuda_check(cudaEventElapsedTime(&ms, ev[s0 + i], ev[s0 + i + 1]), "elapsed time"))
                return -1;
            if (i < max_passes) {
                if (total_ms) total_ms[i] += ms;
                if (launches) launches[i] += 1;
            }
        }
    }
    p->ev_used = 0;  // the events stay in the pool for the next record
    return np;
}

extern "C" const char* sp_last_error(void) { return g_err; }

extern "C" const char* sp_version(void) { return "superpot 0.1 (sm_103a)"; }
