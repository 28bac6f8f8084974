// Autotuner for the stencil kernels: for each launch configuration the
// solvers use (precision, in fixed point or not, mode, fused reduction, dagger,
// right-hand sides) it times every candidate -- register budget (compiler's / capped at 80 for FP32
// and FP16; the fixed-point kernels of FP64 and DF64 have one, and 32, 64 or 128
// threads per block, two a site) x threads per block along the sites, or for the
// multi-RHS kernel x right-hand sides per block (the RHS tile) -- on scratch
// buffers with L2 evicted before each launch, keeps the fastest, and stores
// the choice in a JSON cache keyed by device name, lattice and configuration.
// Launches that have no tuned entry use default_shape (stencil.cu), which is among
// the candidates.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

#include "blas.cuh"

namespace qcd {

// Reads every line of a 256 MB buffer once with ordinary loads: the clean
// lines replace whatever L2 held (twice its size), and dirty lines of earlier
// kernels are written back here, not inside the launch timed next.  The sink
// is written only if the sum equals a value the buffer never produces, which
// keeps the loads.
__global__ void k_l2_evict(const uint4 *__restrict__ buf, size_t n, unsigned *sink)
{
    unsigned acc = 0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const uint4 v = __ldcg(buf + i);
        acc += v.x ^ v.y ^ v.z ^ v.w;
    }
    if (acc == 0x9e3779b9u) *sink = acc;
}

int l2_evict(qcd_ctx *c)
{
    const size_t flush_bytes = 256u << 20;
    int rc;
    if (!c->flush_buf) {
        if ((rc = dev_alloc(c, &c->flush_buf, flush_bytes + 256))) return rc;
        QCD_CUDA_CHECK(cudaMemsetAsync(c->flush_buf, 0x5a, flush_bytes + 256, c->stream));
    }
    c->launches += 1;
    k_l2_evict<<<c->num_sms * 8, 256, 0, c->stream>>>((const uint4 *)c->flush_buf, flush_bytes / sizeof(uint4),
                                                       (unsigned *)((char *)c->flush_buf + flush_bytes));
    QCD_CUDA_CHECK(cudaGetLastError());
    return QCD_OK;
}

namespace {

std::string cache_prefix(qcd_ctx *c)
{
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, c->device) != cudaSuccess) {
        cudaGetLastError();
        std::strcpy(prop.name, "unknown");
    }
    char buf[512];
    std::snprintf(buf, sizeof(buf), "%s|%dx%dx%dx%d|", prop.name, c->g.L[0], c->g.L[1], c->g.L[2], c->g.L[3]);
    return buf;
}

// The cache is a JSON object with one entry per line:
//   "<device>|<Lx>x<Ly>x<Lz>x<Lt>|<key>": [variant, bx, microseconds],
// with "fx|" before the key of a fixed-point kernel (its own bit of it left out)
using Cache = std::map<std::string, qcd_ctx::TuneEntry>;

std::string cache_key(const std::string &prefix, unsigned key)
{
    return prefix + (key & TUNE_KEY_FX ? "fx|" : "") + std::to_string(key & ~TUNE_KEY_FX);
}

// Whether a kernel of configuration s has the shape of a cached entry; another (a
// file written by hand) is timed again.  The kernels exchange values within whole
// warps and hold 384 threads at most, 256 with pipelined hops, 128 in fixed point.
bool shape_ok(const qcd_ctx *c, const StencilCall &s, const qcd_ctx::TuneEntry &e)
{
    if (e.variant < 0 || e.variant > 2) return false;
    if (is_mrhs(s)) return e.bx >= 1 && e.bx <= s.nrhs;
    const bool fx = tune_key(c, s) & TUNE_KEY_FX;
    const int most = fx ? 128 : e.variant == 2 ? 256 : 384;
    return e.bx >= 32 && e.bx % 32 == 0 && e.bx <= most / s.nrhs &&
           (int)nblocks(c->g.Vh, fx ? e.bx / 2 : e.bx) <= c->partial_blocks;
}

Cache read_cache(const char *path)
{
    Cache m;
    if (!path) return m;
    FILE *f = std::fopen(path, "r");
    if (!f) return m;
    char line[1024], key[768];
    while (std::fgets(line, sizeof(line), f)) {
        qcd_ctx::TuneEntry e;
        if (std::sscanf(line, " \"%767[^\"]\" : [ %d , %d , %lf ]", key, &e.variant, &e.bx, &e.us) == 4) m[key] = e;
    }
    std::fclose(f);
    return m;
}

int write_cache(const char *path, const Cache &m)
{
    std::string tmp = std::string(path) + ".tmp";
    FILE *f = std::fopen(tmp.c_str(), "w");
    if (!f) {
        set_error_message("cannot write the tuning cache %s", path);
        return QCD_EINVAL;
    }
    std::fprintf(f, "{\n");
    size_t i = 0;
    for (const auto &kv : m) {
        std::fprintf(f, "  \"%s\": [%d, %d, %.3f]%s\n", kv.first.c_str(), kv.second.variant, kv.second.bx,
                     kv.second.us, ++i < m.size() ? "," : "");
    }
    std::fprintf(f, "}\n");
    std::fclose(f);
    if (std::rename(tmp.c_str(), path) != 0) {
        set_error_message("cannot replace the tuning cache %s", path);
        return QCD_EINVAL;
    }
    return QCD_OK;
}

// scratch: nrhs input and nrhs output vectors of one precision
// the candidates' vectors: in, out and, for one right-hand side, the
// epilogue vector y and the dot operand aux as buffers of their own, so
// that the D^ halves move the bytes they move in a solve
int tune_buffers(qcd_ctx *c, int prec, int nrhs, HVec *in, HVec *out, HVec *y, HVec *aux)
{
    const size_t hb = hvec_bytes(c->g, prec);
    const size_t nb = (size_t)c->g.Vh_pad * sizeof(float);
    const int nv = nrhs == 1 ? 4 : 2;
    const size_t need = nv * nrhs * (hb + nb);
    if (c->tune_bytes < need) {
        if (c->tune_buf) {
            cudaStreamSynchronize(c->stream);
            cudaFree(c->tune_buf);
            for (auto &p : c->pool)
                if (p == c->tune_buf) p = nullptr;
            c->tune_buf = nullptr;
            c->tune_bytes = 0;
        }
        int rc = dev_alloc(c, &c->tune_buf, need);
        if (rc) return rc;
        c->tune_bytes = need;
    }
    char *base = (char *)c->tune_buf;
    HVec *v[4] = {in, out, y, aux};
    for (int k = 0; k < 4; ++k) {
        const int j = k < nv ? k : 0;  // several right-hand sides: y and aux alias in
        v[k]->prec = prec;
        v[k]->p = base + j * nrhs * hb;
        v[k]->norm = (float *)(base + nv * nrhs * hb + j * nrhs * nb);
    }
    // FP64 and DF64 as the solvers run them: fixed-point input
    if (c->fx_links && (prec == QCD_F64 || prec == QCD_DF64)) in->prec = QCD_FX;
    int rc = fill_pattern(c, in->prec, *in, nrhs, hvec_elems(c->g, prec), 11);
    for (int k = 2; k < nv && rc == QCD_OK; ++k) rc = fill_pattern(c, prec, *v[k], nrhs, hvec_elems(c->g, prec), 11 + k);
    return rc;
}

int time_candidate(qcd_ctx *c, const StencilCall &s, double *us)
{
    int rc = QCD_OK;
    cudaEvent_t e0, e1;
    QCD_CUDA_CHECK(cudaEventCreate(&e0));
    QCD_CUDA_CHECK(cudaEventCreate(&e1));
    double best = 1e30;
    for (int it = -1; it < 3; ++it) {
        if ((rc = l2_evict(c))) break;
        QCD_CUDA_CHECK(cudaEventRecord(e0, c->stream));
        if ((rc = launch_stencil(c, s))) break;
        QCD_CUDA_CHECK(cudaEventRecord(e1, c->stream));
        QCD_CUDA_CHECK(cudaEventSynchronize(e1));
        float ms = 0.f;
        QCD_CUDA_CHECK(cudaEventElapsedTime(&ms, e0, e1));
        if (it >= 0 && ms * 1e3 < best) best = ms * 1e3;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc) return rc;
    *us = best;
    return QCD_OK;
}

int tune_one(qcd_ctx *c, StencilCall s, qcd_ctx::TuneEntry *out)
{
    HVec in, o, y, aux;
    int rc = tune_buffers(c, s.prec, s.nrhs, &in, &o, &y, &aux);
    if (rc) return rc;
    s.in = in;
    s.out = o;
    if (in.prec == QCD_FX && s.mode == M_MULT) s.out.prec = QCD_FX;
    s.y = y;
    s.aux = aux;
    s.z = aux;
    s.rhs_stride = hvec_elems(c->g, s.prec);
    s.norm_stride = (size_t)c->g.Vh_pad;
    s.red_args = RedArgs{c->partials, c->counters, c->states + ST_TUNE, FIN_NONE};
    s.done = nullptr;
    // variant 1: the register cap (80 for FP32 and FP16, 128 for DF64);
    // variant 2: the hops software-pipelined (FP32 / FP16 MULT and D^
    // halves, one right-hand side)
    const bool low = s.prec == QCD_F32 || s.prec == QCD_F16;
    const bool pipe = low && s.nrhs == 1 && (s.mode == M_MULT || s.mode == M_DHAT || s.mode == M_FULL);
    const bool mr = is_mrhs(s);
    const int nv = mr ? 2 : pipe ? 3 : (low || (s.prec == QCD_DF64 && !c->fx_links)) ? 2 : 1;
    // sites per block; for the multi-RHS kernel the right-hand sides per block
    // (all, a half, a third, a quarter)
    // (the fixed-point FP64 and DF64 kernels run two threads a site: smaller
    // blocks, and on small lattices the one warp of the default shape)
    const bool fx = in.prec == QCD_FX;
    const bool tiny = fx && (int)nblocks(c->g.Vh, 32) < c->num_sms;
    const int bxs1[] = {64, fx ? 32 : 128, fx ? 16 : 256}, bxsn[] = {32, 64};
    int bxst[4], nt = 0;
    for (int d : {1, 2, 3, 4})
        if (s.nrhs % d == 0) bxst[nt++] = s.nrhs / d;
    const int *bxs = mr ? bxst : s.nrhs > 1 ? bxsn : bxs1;
    const int nbx = mr ? nt : s.nrhs > 1 || (fx && !tiny) ? 2 : 3;
    qcd_ctx::TuneEntry best{0, 128, 1e30};
    // QCD_TUNE_LOG set in the environment: every candidate's time on stderr
    static const bool log = std::getenv("QCD_TUNE_LOG") != nullptr;
    for (int v = 0; v < nv; ++v)
        for (int k = 0; k < nbx; ++k) {
            const int bx = bxs[k];
            if (!mr && bx * s.nrhs > 384) continue;
            if (s.red != R_NONE && (int)nblocks(c->g.Vh, bx) > c->partial_blocks) continue;
            s.force_variant = v;
            s.force_bx = bx;
            double us;
            if ((rc = time_candidate(c, s, &us))) return rc;
            if (log)
                std::fprintf(stderr, "tune prec %d mode %d red %d nrhs %d: variant %d bx %d %.2f us\n", s.prec, s.mode,
                             s.red, s.nrhs, v, fx ? 2 * bx : bx, us);
            if (us < best.us) best = qcd_ctx::TuneEntry{v, fx ? 2 * bx : bx, us};
        }
    *out = best;
    return QCD_OK;
}

}  // namespace

int autotune(qcd_ctx *c, const char *cache_path)
{
    if (!c->have_clover) {
        set_error_message("qcd_autotune needs the gauge field and the clover term");
        return QCD_ESTATE;
    }
    struct Cfg {
        int prec, mode, red, nrhs;
    };
    const Cfg cfgs[] = {
        {QCD_F64, M_MULT, R_NONE, 1},  {QCD_F64, M_DHAT, R_DOT_AUX, 1}, {QCD_F64, M_DHAT, R_OMEGA, 1},
        {QCD_F64, M_SRC, R_NONE, 1},   {QCD_F64, M_FULL, R_NORM, 1},    {QCD_F64, M_DHAT, R_NORM, 1},
        {QCD_F32, M_MULT, R_NONE, 1},  {QCD_F32, M_DHAT, R_DOT_AUX, 1}, {QCD_F32, M_DHAT, R_OMEGA, 1},
        {QCD_F32, M_HOP, R_NONE, 1},   {QCD_F32, M_MULT, R_NONE, 12},  {QCD_F32, M_HOP, R_NONE, 12},
        {QCD_F16, M_MULT, R_NONE, 1},  {QCD_F16, M_DHAT, R_DOT_AUX, 1}, {QCD_F16, M_DHAT, R_OMEGA, 1},
        {QCD_F16, M_MULT, R_NONE, 12},
        {QCD_DF64, M_MULT, R_NONE, 1}, {QCD_DF64, M_DHAT, R_DOT_AUX, 1}, {QCD_DF64, M_DHAT, R_OMEGA, 1},
        {QCD_DF64, M_SRC, R_NONE, 1},  {QCD_DF64, M_DHAT, R_NORM, 1},
        // the second halves of the gamma5-hermitian S_ee
        {QCD_F64, M_FULL, R_DOT_AUX, 1}, {QCD_F64, M_FULL, R_OMEGA, 1},
        {QCD_F32, M_FULL, R_DOT_AUX, 1}, {QCD_F32, M_FULL, R_OMEGA, 1},
        {QCD_F16, M_FULL, R_DOT_AUX, 1}, {QCD_F16, M_FULL, R_OMEGA, 1},
        {QCD_DF64, M_FULL, R_DOT_AUX, 1}, {QCD_DF64, M_FULL, R_OMEGA, 1}, {QCD_DF64, M_FULL, R_NORM, 1},
    };
    Cache cache = read_cache(cache_path);
    const std::string prefix = cache_prefix(c);
    bool changed = false;
    const bool prof = c->profiling;
    c->profiling = false;
    int rc = QCD_OK;
    for (const Cfg &f : cfgs) {
        StencilCall s;
        s.prec = f.prec;
        s.mode = f.mode;
        s.red = f.red;
        s.nrhs = f.nrhs;
        s.out_par = 0;
        s.a = 1.0;
        s.cc = -c->kappa * c->kappa;
        const unsigned key = tune_key(c, s);
        const std::string ck = cache_key(prefix, key);
        auto hit = cache.find(ck);
        if (hit != cache.end() && shape_ok(c, s, hit->second)) {
            c->tune[key] = hit->second;
            continue;
        }
        qcd_ctx::TuneEntry e;
        if ((rc = tune_one(c, s, &e))) break;
        c->tune[key] = e;
        cache[ck] = e;
        changed = true;
    }
    c->profiling = prof;
    if (rc) return rc;
    if (cache_path && changed) return write_cache(cache_path, cache);
    return QCD_OK;
}

int tune_entries(qcd_ctx *c, int max, unsigned *keys, int *variant, int *bx, double *us)
{
    int n = 0;
    for (const auto &kv : c->tune) {
        if (n < max) {
            if (keys) keys[n] = kv.first & ~TUNE_KEY_FX;
            if (variant) variant[n] = kv.second.variant;
            if (bx) bx[n] = kv.second.bx;
            if (us) us[n] = kv.second.us;
        }
        ++n;
    }
    return n;
}

}  // namespace qcd
