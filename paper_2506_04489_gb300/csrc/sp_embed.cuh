// Solve passes for grids whose padded length 2n has no plan of its own: the same five
// passes on transform lengths F >= 2n that have one.
//
// The solve is the aperiodic convolution u_i = sum_j K_{i-j} rho_j, |i - j| <= n - 1, with
// K = IDFT_{2n}(M) per axis (real and even).  Its cyclic form holds for every period
// F >= 2n - 1, so the plan keeps the multiplier of period F (built once from the 2n one,
// sp_setup.cu), and the passes zero-pad to F and crop to n.  Nothing is approximated: the
// results differ from the 2n transforms by rounding alone.  A prime n costs what its
// neighbours do, where transforms of its own length need Bluestein's algorithm.
//
// The kernels are those of sp_v2.cuh with a bound on the line's grid points (RAG): rows at
// and above n are zero on input and not written on output.  Measured at n = 101 (double-
// float): 171 us; the runtime-radix passes of sp_passes.cu took 1.17 ms.
#pragma once

#include "sp_v2.cuh"

namespace v2 {

// Largest tile (columns) and the register cap, as resident CTAs of that size: 16-byte types
// run E = 12 and above at 168 registers (spilling below it costs 10 to 40 %; 128 where a
// line has 64 threads or more), fewer values at 128 (96 for E = 6); 8-byte types at 64, 96
// or 128 by E.  CTAs of 8-byte types go up to 512 threads, so that lines of 33 to 64 threads
// keep tiles of 8 columns, 64 contiguous bytes a row (x / y forward / y inverse, us, 4 columns
// against 8: 210^3 (F = 432) 224/72/80 / 177/59/67, 285^3 (576) 558/166/191 / 446/142/172).
// Double-float passes of one transform on eight values and 32 threads or more a line are light:
// 96 registers hold them (y forward/inverse, z forward/inverse, us, 128 against 96: 150^3 70/73,
// 59/54 / 66/68, 55/49; 300^3 599/639, 401/401 / 587/578, 346/345 with tiles of 4 columns on 320
// threads; the x pass spills and loses 5 to 10 %).
template <class R, class K, int N, int MODE> constexpr bool rag_light()
{
    return std::is_same<R, df32>::value && PlanOf<K, N>::E <= 8 && N / PlanOf<K, N>::E >= 32 && MODE != XMUL;
}
template <class R, int N, int MODE> constexpr int rag_b_max()
{
    constexpr int T = N / PlanOf<R, N>::E;
    int b = sizeof(cpx<R>) >= 16 && T >= 32 ? 4 : 16;  // the most that rag_tile takes
    while (b > 2 && b * T > (sizeof(cpx<R>) < 16 ? 512 : (rag_light<R, R, N, MODE>() ? 320 : 256))) b /= 2;
    return b;
}
template <class R, class K, int N, int MODE> constexpr int rag_min_blocks(int threads)
{
    constexpr int E = PlanOf<K, N>::E, T = N / E;
    constexpr int cap = sizeof(cpx<R>) >= 16 ? (E <= 6 || rag_light<R, K, N, MODE>() ? 96 : (E >= 12 && T < 64 ? 168 : 128)) : (E <= 8 ? 64 : (E <= 16 ? 96 : 128));
    const int b = 65536 / (cap * threads);
    return b < 1 ? 1 : b;
}

template <class R, int N, int MODE>
__global__ void __launch_bounds__((N / PlanOf<R, N>::E) * rag_b_max<R, N, MODE>(),
                                  rag_min_blocks<R, R, N, MODE>((N / PlanOf<R, N>::E) * rag_b_max<R, N, MODE>())) k_rag_line(LArgs a)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    grid_dependency();
    line_tile<R, N, MODE, -1, R, true>(a, blockIdx.x, a.reverse ? gridDim.y - 1 - blockIdx.y : blockIdx.y, blockIdx.z, smraw);
}

template <class R, int N> constexpr int rag_pairs_max()
{
    constexpr int T = N / PlanOf<ZKey<R>, N>::E;
    return T >= 128 ? 1 : 128 / T;
}
template <class R, class Tio, int N, bool FORWARD>
__global__ void __launch_bounds__((N / PlanOf<ZKey<R>, N>::E) * rag_pairs_max<R, N>(),
                                  rag_min_blocks<R, ZKey<R>, N, FWD>((N / PlanOf<ZKey<R>, N>::E) * rag_pairs_max<R, N>()))
    k_rag_z(ZArgs2 a)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    grid_dependency();
    const int blk = a.reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    if constexpr (FORWARD) zf_tile<R, Tio, N, true>(a, blk, blockIdx.y, smraw);
    else zi_tile<R, Tio, N, true>(a, blk, blockIdx.y, smraw);
}

// Columns of a CTA of a line pass: 8 (128 bytes of a row at 16-byte values), 4 where a line
// has 32 threads or more (smaller CTAs wait less at their barriers: double-float at 320 to
// 768 4 to 12 % faster than 8; 2 loses more to half-used sectors), more where a line has
// fewer than eight threads; halved while that leaves fewer than two CTAs on each of 152 SMs.
template <class R, int N> int rag_tile(int T, int bmax, long long columns, long long outer)
{
    int b = T >= 32 && sizeof(cpx<R>) >= 16 ? 4 : 8;
    while (T * b < 64) b *= 2;
    if (b > bmax) b = bmax;
    while (b > 2 && T * b > 32 && (columns + b - 1) / b * outer < 304) b /= 2;
    return b;
}
// Pairs of lines of a CTA of a z pass: whole warps as nearly as they come, 64 to 128 threads.
inline int rag_pairs(int T, int bmax, long long pairs)
{
    int best = 1;
    double use = 0.0;
    for (int b = 1; b <= bmax && (b == 1 || T * b <= 128); ++b) {
        const double u = (double)(T * b) / ((T * b + 31) / 32 * 32) * (T * b < 64 ? 0.9 : 1.0);
        if (u >= use) {
            use = u;
            best = b;
        }
    }
    while (best > 1 && T * best > 32 && (pairs + best - 1) / best < 304) best = (best + 1) / 2;
    return best;
}

// FP32 y passes that run the pipelined kernel (k3_line): they move a row in and half a row out,
// or the reverse, with one transform between, so what bounds them is the latency of the loads,
// which the pipeline takes out.  Inverse passes load whole rows and gain from F = 256 up
// (us, plain tile against pipeline: 125^3 16.4 / 13.8, 200^3 66 / 41, 250^3 144 / 74, 285^3
// 172 / 144), forward passes, whose loads are half as many, from 400 (200^3 47 / 41, 250^3
// 102 / 72; 240x180x75 24.8 / 26.7).  Few tiles leave the persistent CTAs without a next one to
// load (39x172x122, 1326 tiles, three a CTA: 3 % slower; 240x180x75, 2640: 2 % faster): from 16
// an SM (152 of them).  Eight values a thread have warps enough without it, and the x pass
// computes twice as long a byte (200^3 117 / 144).  Above 864 all but the forward pass at 1280
// need more than 110 KB; that one would gain (100x600x100 64 / 56, 200x640x100 131 / 101) and
// is left on the plain tile.
constexpr long long kPipeTiles = 16 * 152;
template <class R, int N, int MODE> constexpr bool rag_pipe()
{
    return std::is_same<R, float>::value && PlanOf<R, N>::E >= 12 &&
           N <= 864 &&
           (MODE == INV ? N >= 256 : MODE == FWD && N >= 400) && pipe_smem<R, N, MODE, R, true>() <= 110 * 1024;
}
template <class R, int N, int MODE> sp_status rag_line(const LArgs& a, int outer, int batch, cudaStream_t st)
{
    constexpr int T = N / PlanOf<R, N>::E;
    LArgs ab = a;
    if constexpr (rag_pipe<R, N, MODE>()) {
        constexpr int B = 1 << lg_default<N>();
        if ((long long)((a.ncol + B - 1) / B) * outer * batch >= kPipeTiles && pipe_fits<R, N, MODE, R, true>(a)) {
            ab.B = B;
            ab.lgB = lg_default<N>();
            return launch_pipe<R, N, MODE, R, true>(ab, outer, batch, st);
        }
    }
    ab.B = rag_tile<R, N>(T, rag_b_max<R, N, MODE>(), a.ncol, (long long)outer * batch);
    ab.lgB = 0;
    while ((1 << ab.lgB) < ab.B) ++ab.lgB;
    const size_t smem = line_smem<R, N, MODE>(ab.B);
    sp_status rc;
    if ((rc = smem_attr<k_rag_line<R, N, MODE>>(smem))) return rc;
    dim3 grid((unsigned)((a.ncol + ab.B - 1) / ab.B), (unsigned)outer, (unsigned)batch);
    return launch_pass(k_rag_line<R, N, MODE>, grid, T * ab.B, smem, st, ab, a.dependent != 0, "ragged line pass");
}

template <class R, class Tio, int N> sp_status rag_z(const ZArgs2& a, bool forward, int batch, cudaStream_t st)
{
    constexpr int T = N / PlanOf<ZKey<R>, N>::E;
    ZArgs2 ab = a;
    const long long pairs = (a.lines + 1) / 2;
    ab.B = rag_pairs(T, rag_pairs_max<R, N>(), pairs * batch);
    const size_t smem = pass_tw_bytes<R, N, ZKey<R>>() + sizeof(cpx<R>) * (z_two_buffers<R, N>(ab.B) ? 2 : 1) * z_buf<R, N>(ab.B);
    dim3 grid((unsigned)((pairs + ab.B - 1) / ab.B), (unsigned)batch);
    sp_status rc;
    if (forward) {
        if ((rc = smem_attr<k_rag_z<R, Tio, N, true>>(smem))) return rc;
        return launch_pass(k_rag_z<R, Tio, N, true>, grid, T * ab.B, smem, st, ab, a.dependent != 0, "ragged z forward pass");
    } else {
        if ((rc = smem_attr<k_rag_z<R, Tio, N, false>>(smem))) return rc;
        return launch_pass(k_rag_z<R, Tio, N, false>, grid, T * ab.B, smem, st, ab, a.dependent != 0, "ragged z inverse pass");
    }
}

// Calls f.template run<F>() for a listed length F.
template <class Fn> inline sp_status with_f(int F, Fn&& f)
{
    switch (F) {
#define SP_F_CASE(L) \
    case L: return f.template run<L>();
        SP_F_LENGTHS(SP_F_CASE)
#undef SP_F_CASE
        default: return SP_ERR_UNSUPPORTED_SIZE;
    }
}
template <class R, int MODE> struct RagLineRun {
    const LArgs* a;
    int outer, batch;
    cudaStream_t st;
    template <int F> sp_status run() { return rag_line<R, F, MODE>(*a, outer, batch, st); }
};
template <class R, class Tio> struct RagZRun {
    const ZArgs2* a;
    bool forward;
    int batch;
    cudaStream_t st;
    template <int F> sp_status run() { return rag_z<R, Tio, F>(*a, forward, batch, st); }
};
template <class R> struct RagRadices {
    int* out;
    bool z;
    template <int F> sp_status run()
    {
        if (z) copy_radices<ZKey<R>, F>(out);
        else copy_radices<R, F>(out);
        return SP_OK;
    }
};

// Axes whose own padded length has a tuned plan keep it (their tables are N's).
inline bool own_plan(const sp_plan p, int ax) { return p->d_twF[ax] == nullptr; }
template <class R> const void* embed_tw(sp_plan p, int ax) { return own_plan(p, ax) ? Tabs<R>::tw(p, ax) : p->d_twF[ax]; }

template <class R, int MODE> sp_status embed_line(sp_plan p, int ax, const LArgs& a, int outer, int batch, cudaStream_t st)
{
    if (own_plan(p, ax)) return with_len(p->F[ax], LineRun<R, MODE>{&a, outer, batch, st, 0});
    return with_f(p->F[ax], RagLineRun<R, MODE>{&a, outer, batch, st});
}
template <class R, class Tio> sp_status embed_z(sp_plan p, const ZArgs2& a, bool forward, int batch, cudaStream_t st)
{
    if (own_plan(p, 2)) return with_len(p->F[2], ZRun<R, Tio>{&a, forward, batch, st});
    return with_f(p->F[2], RagZRun<R, Tio>{&a, forward, batch, st});
}

// The whole solve on the lengths F (the schedule of v2::solve).
template <class R, class Tio> sp_status solve_embed(sp_plan p, const void* rho, void* u, int batch, cudaStream_t st)
{
    p->npass = 5;
    p->pass_name[0] = "z_forward";
    p->pass_name[1] = "y_forward";
    p->pass_name[2] = "x_multiply";
    p->pass_name[3] = "y_inverse";
    p->pass_name[4] = "z_inverse";
    ZArgs2 z = {};
    z.rho = rho;
    z.u = u;
    z.W = p->d_work;
    z.n1 = p->n[1];
    z.n2 = p->n[2];
    z.lines = (long long)p->n[0] * p->n[1];
    z.plane = p->planef;
    z.ldz = p->ldf;
    z.io_bs = (long long)p->n[0] * p->n[1] * p->n[2];
    z.w_bs = (long long)p->n[0] * p->planef;
    z.tw = embed_tw<R>(p, 2);
    z.dependent = (size_t)batch * z.w_bs * sizeof(cpx<R>) <= kDependentBytes;
    LArgs y = {};
    y.in = y.out = p->d_work;
    y.in_os = y.out_os = p->planef;
    y.in_es = y.out_es = p->ldf;
    y.in_bs = y.out_bs = z.w_bs;
    y.ncol = p->F[2] / 2 + 1;
    y.in_ld = p->ldf;
    y.tw = embed_tw<R>(p, 1);
    y.nlim = p->n[1];
    y.dependent = z.dependent;
    LArgs x = y;
    x.in_os = x.out_os = p->ldf;
    x.in_es = x.out_es = p->planef;
    x.tw = embed_tw<R>(p, 0);
    x.M = p->d_Ms;
    x.No = p->F[1];
    x.nh_line = p->F[0] / 2;
    x.ldzM = p->ldf;
    x.nlim = p->n[0];
    LArgs yf = y;
    yf.reverse = 1;
    ZArgs2 zi = z;
    zi.reverse = 1;
    sp_status rc;
    if ((rc = sp_mark(p, st))) return rc;
    if ((rc = embed_z<R, Tio>(p, z, true, batch, st))) return rc;
    if ((rc = sp_mark(p, st))) return rc;
    if ((rc = embed_line<R, FWD>(p, 1, yf, p->n[0], batch, st))) return rc;
    if ((rc = sp_mark(p, st))) return rc;
    if ((rc = embed_line<R, XMUL>(p, 0, x, p->F[1], batch, st))) return rc;
    if ((rc = sp_mark(p, st))) return rc;
    if ((rc = embed_line<R, INV>(p, 1, y, p->n[0], batch, st))) return rc;
    if ((rc = sp_mark(p, st))) return rc;
    if ((rc = embed_z<R, Tio>(p, zi, false, batch, st))) return rc;
    return sp_mark(p, st);
}

// Staged twiddle tables of the axes that run a length F of their own (the base twiddles of
// F are in place).
template <class R> sp_status embed_twiddles(sp_plan p, cudaStream_t st)
{
    for (int ax = 0; ax < 3; ++ax) {
        if (own_plan(p, ax)) continue;
        cpx<R>* tw = static_cast<cpx<R>*>(p->d_twF[ax]);
        const sp_status rc = ax == 2 ? with_f(p->F[ax], StageTw<R, ZKey<R>>{tw, st}) : with_f(p->F[ax], StageTw<R, R>{tw, st});
        if (rc) return rc;
    }
    return SP_OK;
}
template <class R> sp_status embed_radices(sp_plan p, int* out)
{
    for (int ax = 0; ax < 3; ++ax)
        if (const sp_status rc = with_f(p->F[ax], RagRadices<R>{out + 8 * ax, ax == 2})) return rc;
    return SP_OK;
}

}  // namespace v2

// Explicit instantiation of the passes of one length, so that they compile in translation
// units of their own (PREFIX = extern to declare).
#define SP_EMBED_LINES(PREFIX, R, L)                                                         \
    PREFIX template sp_status v2::rag_line<R, L, v2::FWD>(const v2::LArgs&, int, int, cudaStream_t); \
    PREFIX template sp_status v2::rag_line<R, L, v2::INV>(const v2::LArgs&, int, int, cudaStream_t); \
    PREFIX template sp_status v2::rag_line<R, L, v2::XMUL>(const v2::LArgs&, int, int, cudaStream_t);
#define SP_EMBED_Z(PREFIX, R, Tio, L) PREFIX template sp_status v2::rag_z<R, Tio, L>(const v2::ZArgs2&, bool, int, cudaStream_t);
#define SP_EMBED_FLOAT(PREFIX, L) SP_EMBED_LINES(PREFIX, float, L) SP_EMBED_Z(PREFIX, float, float, L) SP_EMBED_Z(PREFIX, float, double, L)
#define SP_EMBED_DOUBLE(PREFIX, L) SP_EMBED_LINES(PREFIX, double, L) SP_EMBED_Z(PREFIX, double, double, L)
#define SP_EMBED_DF32(PREFIX, L) SP_EMBED_LINES(PREFIX, df32, L) SP_EMBED_Z(PREFIX, df32, double, L)
// The lengths in four groups of about equal compile time.
#define SP_F_GROUP1(X, PREFIX) X(PREFIX, 16) X(PREFIX, 32) X(PREFIX, 48) X(PREFIX, 200) X(PREFIX, 384) X(PREFIX, 432) X(PREFIX, 2048)
#define SP_F_GROUP2(X, PREFIX) X(PREFIX, 64) X(PREFIX, 72) X(PREFIX, 80) X(PREFIX, 216) X(PREFIX, 320) X(PREFIX, 512) X(PREFIX, 1280)
#define SP_F_GROUP3(X, PREFIX) X(PREFIX, 96) X(PREFIX, 128) X(PREFIX, 144) X(PREFIX, 400) X(PREFIX, 576) X(PREFIX, 864) X(PREFIX, 1024)
#define SP_F_GROUP4(X, PREFIX) X(PREFIX, 160) X(PREFIX, 192) X(PREFIX, 256) X(PREFIX, 288) X(PREFIX, 640) X(PREFIX, 768) X(PREFIX, 1536)
