// kg_ensemble.cu -- C ABI of the batched parametric ensemble (kg_ens_*).
//
// Many independent instances of the scheme of section 1.1.2 (Eq. (2)) on 64^3 and
// 128^3 grids, initial data u0 = A exp(-|x|^2 / s^2), v0 = 0 (the parametric blow-up
// studies of section 1), advanced together: up to kLaunchSteps time steps of the whole
// ensemble are one persistent cooperative launch (k_ens_run).  Launch shape (CTAs per SM, unit visiting order) comes from a small
// autotuner that times the candidates on the actual ensemble.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/kg.h"
#include "kg_ensemble.cuh"
#include "kg_launch.h"

using namespace kg;

namespace kg {
__global__ void __launch_bounds__(128) k_ens_axis(const EnsInst* inst, const double* s, double L, const double2* tw64,
                                                  const double2* tw128, EnsAxis* out) {
    __shared__ double g[128], g3[128];
    const int i = blockIdx.x, t = threadIdx.x, N = inst[i].N;
    const double2* tw = N == 64 ? tw64 : tw128;   // exp(-2 pi i j / N)
    EnsAxis& ax = out[i];
    if (t < N) {
        const double x = -L / 2 + (L / N) * t;
        const double v = exp(-x * x * (1.0 / (s[i] * s[i])));
        g[t] = v;
        g3[t] = v * v * v;
        ax.g[t] = v;
    }
    __syncthreads();
    if (t <= N / 2) {
        NSum a, b;
        a.s = a.c = b.s = b.c = 0.0;
        for (int j = 0; j < N; j++) {
            const double c = tw[(t * j) & (N - 1)].x;
            a.add(g[j] * c);
            b.add(g3[j] * c);
        }
        ax.G[t] = a.value();
        ax.G3[t] = b.value();
    }
}
}  // namespace kg

namespace {

constexpr int kLaunchSteps = 50;   // steps of one launch, and between looks at the blow-up flags

// Units drawn at a time.  Drawing costs about 2 us of one thread's dependent loads and fences,
// against 5 to 10 us of work in a unit, so runs of several pay, as long as a pass keeps about three
// runs for every CTA (else they wait for the slowest of the pass before).  ms per step with runs of
// 1, 2, 4, 8: 48 + 48 instances double-float 3.02, 2.83, 2.74, 2.73; 256 x 64^3 FP32 1.06, 0.89,
// 0.81, 0.79; 48 + 48 FP32 1.78, 1.47, 1.33, 1.31.
constexpr int kMostRun = 8;

// y or z units of a pass over n64 and n128 instances (in the double-float tile width)
constexpr int pass_units(int n64, int n128) { return 80 * n64 + 576 * n128; }

// launch shape chosen by kg_ens_tune, reused by later kg_ens_init calls with the
// same precision and the same numbers of 64^3 and 128^3 instances (in this process, and
// through the cache file of kg_ens_set_tune_cache in later ones)
struct Tuned {
    bool valid = false;
    int prec = 0, n64 = 0, n128 = 0, sched = 0, bps = 2, order = 1;
};
Tuned g_tuned;
std::string g_cache_path;   // kg_ens_set_tune_cache ("" = no file)

int efail(int code, const std::string& msg);

// the device the cache entries are keyed by: name (spaces as '_') and SM count
std::string device_key() {
    int dev = 0, sms = 0;
    cudaDeviceProp prop;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return "unknown";
    sms = prop.multiProcessorCount;
    std::string name = prop.name;
    for (char& ch : name)
        if (ch == ' ' || ch == '\t') ch = '_';
    return name + " " + std::to_string(sms);
}

// cache file: one line per key, "kgens <prec> <n64> <n128> <device> <sms> <sched> <bps> <order> <ms>"
bool cache_lookup(int prec, int n64, int n128, Tuned* out) {
    if (g_cache_path.empty()) return false;
    FILE* f = std::fopen(g_cache_path.c_str(), "r");
    if (!f) return false;
    const std::string dk = device_key();
    char line[512];
    bool found = false;
    while (std::fgets(line, sizeof(line), f)) {
        char tag[16], dname[256];
        int pr, a, b, sms, sc, bp, od;
        double ms;
        if (std::sscanf(line, "%15s %d %d %d %255s %d %d %d %d %lf", tag, &pr, &a, &b, dname, &sms, &sc, &bp, &od,
                        &ms) != 10)
            continue;
        if (std::string(tag) != "kgens" || pr != prec || a != n64 || b != n128) continue;
        if (std::string(dname) + " " + std::to_string(sms) != dk) continue;
        if (sc < 0 || sc >= kEnsSchedules || bp < 1 || (od != 0 && od != 1)) continue;
        out->valid = true;
        out->prec = prec;
        out->n64 = n64;
        out->n128 = n128;
        out->sched = sc;
        out->bps = bp;
        out->order = od;
        found = true;
    }
    std::fclose(f);
    return found;
}

// replace (or add) the entry of t in the cache file; the file is rewritten through a
// temporary file and a rename, so a reader never sees half of it
int cache_store(const Tuned& t, double ms) {
    if (g_cache_path.empty()) return KG_OK;
    std::vector<std::string> keep;
    const std::string dk = device_key();
    if (FILE* f = std::fopen(g_cache_path.c_str(), "r")) {
        char line[512];
        while (std::fgets(line, sizeof(line), f)) {
            char tag[16], dname[256];
            int pr, a, b, sms;
            const bool parsed = std::sscanf(line, "%15s %d %d %d %255s %d", tag, &pr, &a, &b, dname, &sms) == 6;
            const bool same = parsed && std::string(tag) == "kgens" && pr == t.prec && a == t.n64 && b == t.n128 &&
                              std::string(dname) + " " + std::to_string(sms) == dk;
            if (!same) keep.push_back(line);
        }
        std::fclose(f);
    }
    const std::string tmp = g_cache_path + ".tmp";
    FILE* f = std::fopen(tmp.c_str(), "w");
    if (!f) return efail(KG_EINVAL, "cannot write the tune cache " + tmp);
    for (const auto& l : keep) std::fputs(l.c_str(), f);
    std::fprintf(f, "kgens %d %d %d %s %d %d %d %.4f\n", t.prec, t.n64, t.n128, dk.c_str(), t.sched, t.bps, t.order,
                 ms);
    const bool ok = std::fclose(f) == 0;
    if (!ok || std::rename(tmp.c_str(), g_cache_path.c_str()) != 0)
        return efail(KG_EINVAL, "cannot replace the tune cache " + g_cache_path);
    return KG_OK;
}

void count_sizes(const std::vector<int>& Ns, int* n64, int* n128) {
    *n64 = 0;
    *n128 = 0;
    for (int n : Ns) (n == 64 ? *n64 : *n128) += 1;
}

int efail(int code, const std::string& msg) { return set_last_error(code, msg); }

#define KG_ECK(call)                                                                               \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess) return efail(KG_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

// low-mode shell energies of uh^0: (h^3/N^3) sum_{shell} w_k omega_k^2 |uh_k|^2 / 2,
// shells |m| in {0}, (0,1], (1,2], (2,4]; one CTA per instance
template <int N>
__device__ __forceinline__ void shells(const double2* __restrict__ uh, int lg, double L, double* __restrict__ out4) {
    __shared__ double acc[4][256];
    double loc[4] = {0, 0, 0, 0};
    const double kf = 2.0 * 3.14159265358979323846 / L;
    for (int t = threadIdx.x; t < 9 * 9 * 5; t += blockDim.x) {   // |m| <= 4 box, kx >= 0
        const int mx = t % 5, my = (t / 5) % 9 - 4, mz = t / 45 - 4;
        const int m2 = mx * mx + my * my + mz * mz;
        const int sh = (m2 == 0) ? 0 : (m2 <= 1) ? 1 : (m2 <= 4) ? 2 : (m2 <= 16) ? 3 : -1;
        if (sh < 0) continue;
        const int ky = (my + N) % N, kz = (mz + N) % N;
        const double2 v = uh[Lay<N>::zcol(ky, mx, lg) + ((size_t)kz << lg)];
        const double w = (mx == 0 || mx == N / 2) ? 1.0 : 2.0;
        loc[sh] += w * 0.5 * (1.0 + kf * kf * m2) * (v.x * v.x + v.y * v.y);
    }
    for (int q = 0; q < 4; q++) acc[q][threadIdx.x] = loc[q];
    __syncthreads();
    if (threadIdx.x < 4) {
        double s = 0.0;
        for (int i = 0; i < 256; i++) s += acc[threadIdx.x][i];
        const double h = L / N;
        out4[threadIdx.x] = s * h * h * h / ((double)N * N * N);
    }
}

__global__ void __launch_bounds__(256) k_shells(const EnsInst* inst, int lg, double L, double* out) {
    const EnsInst& in = inst[blockIdx.x];
    if (in.N == 64) shells<64>(in.S0, lg, L, out + 4 * blockIdx.x);
    else shells<128>(in.S0, lg, L, out + 4 * blockIdx.x);
}

// shell energies of many sampled Gaussians A exp(-|x|^2/s^2) on the N^3 grid: the field
// is a product g(x) g(y) g(z), so its low modes are A G(mx) G(my) G(mz) with G the 1D DFT
// of g; one thread per point, same shells and weights as k_shells
__global__ void k_gauss_shells(int count, int N, double L, const double* __restrict__ A,
                               const double* __restrict__ S, double* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const double h = L / N, inv_s2 = 1.0 / (S[i] * S[i]);
    double gr[5] = {0, 0, 0, 0, 0}, gi[5] = {0, 0, 0, 0, 0};   // G(m), m = 0..4 (G(-m) = conj G(m))
    for (int j = 0; j < N; j++) {
        const double x = -L / 2 + h * j;
        const double gv = exp(-x * x * inv_s2);
        for (int m = 0; m < 5; m++) {
            double sn, cs;
            sincospi(-2.0 * (double)((m * j) % N) / (double)N, &sn, &cs);
            gr[m] += gv * cs;
            gi[m] += gv * sn;
        }
    }
    double acc[4] = {0, 0, 0, 0};
    const double kf = 2.0 * 3.14159265358979323846 / L;
    for (int mz = -4; mz <= 4; mz++)
        for (int my = -4; my <= 4; my++)
            for (int mx = 0; mx <= 4; mx++) {
                const int m2 = mx * mx + my * my + mz * mz;
                const int sh = (m2 == 0) ? 0 : (m2 <= 1) ? 1 : (m2 <= 4) ? 2 : (m2 <= 16) ? 3 : -1;
                if (sh < 0) continue;
                const int ay = my < 0 ? -my : my, az = mz < 0 ? -mz : mz;
                // |G(mx) G(my) G(mz)|^2 = |G(mx)|^2 |G(|my|)|^2 |G(|mz|)|^2
                const double p = (gr[mx] * gr[mx] + gi[mx] * gi[mx]) * (gr[ay] * gr[ay] + gi[ay] * gi[ay]) *
                                 (gr[az] * gr[az] + gi[az] * gi[az]);
                const double w = (mx == 0) ? 1.0 : 2.0;
                acc[sh] += w * 0.5 * (1.0 + kf * kf * m2) * A[i] * A[i] * p;
            }
    const double norm = h * h * h / ((double)N * N * N);
    for (int q = 0; q < 4; q++) out[4 * (size_t)i + q] = acc[q] * norm;
}

struct Ens {
    int count = 0, prec = KG_DF64;
    double L = 0, dt = 0, lam = 1.0;
    std::vector<int> Ns;
    Tables tab[2];              // [0]: 64^3, [1]: 128^3
    bool have[2] = {false, false};
    std::vector<void*> allocs;
    size_t bytes = 0;
    std::vector<EnsInst> h_inst;
    EnsInst* d_inst = nullptr;
    EnsPlan* d_plan = nullptr;
    int* d_status = nullptr;
    int* d_order = nullptr;
    double* d_feat = nullptr;
    double2* tmp = nullptr;     // two FP64 spectral scratch arrays of the largest grid
    double2* tmp2 = nullptr;
    double* phys = nullptr;     // physical scratch of the largest grid
    cudaStream_t stream = nullptr;
    const PassLaunch* pl = nullptr;
    int bps = 1, grid = 0, order = 0, nsm = 0, sched = 0;
    double threshold = -1.0;
    int missing = 0;
    long long spin_limit = 1ll << 24;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
};

Ens* g_ens = nullptr;

int ealloc(Ens* e, void** p, size_t bytes, const char* what) {
    cudaError_t r = cudaMalloc(p, bytes);
    if (r != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        return efail(KG_ENOMEM, std::string("cudaMalloc(") + what + "): " + cudaGetErrorString(r));
    }
    e->allocs.push_back(*p);
    e->bytes += bytes;
    return KG_OK;
}

void ens_destroy(Ens* e) {
    if (!e) return;
    if (e->stream) cudaStreamSynchronize(e->stream);
    for (void* p : e->allocs) cudaFree(p);
    if (e->ev0) cudaEventDestroy(e->ev0);
    if (e->ev1) cudaEventDestroy(e->ev1);
    if (e->stream) cudaStreamDestroy(e->stream);
    delete e;
}

unsigned threshold_key(double thr) {
    if (!(thr > 0.0)) return 0xFFFFFFFFu;
    float f = (float)thr;
    unsigned k;
    std::memcpy(&k, &f, 4);
    return k;
}

EnsParams make_params(const Ens* e) {
    EnsParams p;
    std::memset(&p, 0, sizeof(p));
    p.inst = e->d_inst;
    p.count = e->count;
    p.plan = e->d_plan;
    for (int t = 0; t < 2; t++) {
        if (e->have[t]) {
            p.tab[t].tw = e->tab[t].tw;
            p.tab[t].coef = e->tab[t].coef;
        }
    }
    p.status = e->d_status;
    p.order_idx = e->d_order;
    p.lam = e->lam;
    p.thr_key = threshold_key(e->threshold);
    p.run = kMostRun;
    p.missing = e->missing;
    p.spin_limit = e->spin_limit;
    return p;
}

int upload_order(Ens* e) {
    std::vector<int> idx(e->count);
    for (int i = 0; i < e->count; i++) idx[i] = i;
    if (e->order == 1)   // larger grids first
        std::stable_sort(idx.begin(), idx.end(), [e](int a, int b) { return e->Ns[a] > e->Ns[b]; });
    KG_ECK(cudaMemcpy(e->d_order, idx.data(), sizeof(int) * e->count, cudaMemcpyHostToDevice));
    return KG_OK;
}

int check_status(Ens* e) {
    int st = 0;
    KG_ECK(cudaMemcpy(&st, e->d_status, sizeof(int), cudaMemcpyDeviceToHost));
    if (st != 0) return efail(KG_ETIMEOUT, "a bounded wait of the ensemble kernel gave up");
    return KG_OK;
}

int set_shape(Ens* e, int sched, int bps, int order) {
    const int maxb = e->pl->ens_blocks_per_sm(sched);
    if (maxb < 1) return efail(KG_ECUDA, "ensemble kernel cannot be resident (occupancy 0)");
    e->sched = sched;
    e->bps = std::max(1, std::min(bps, maxb));
    e->grid = e->bps * e->nsm;
    e->order = order;
    return upload_order(e);
}

// n steps of every live instance, in launches of at most kLaunchSteps
int launch_steps(Ens* e, int n) {
    const EnsParams p = make_params(e);
    for (; n > 0; n -= kLaunchSteps) {
        KG_ECK(e->pl->ens_run(p, e->grid, e->sched, e->order, std::min(n, kLaunchSteps), e->stream));
    }
    return KG_OK;
}

}  // namespace

extern "C" {

int kg_ens_init(int count, const int* Ns, double L, double dt, const double* A, const double* s) {
    if (count < 1 || count > kEnsMaxInst) return efail(KG_EINVAL, "count must be in [1, 1024]");
    if (!Ns || !A || !s) return efail(KG_EINVAL, "NULL argument");
    if (!(L > 0.0) || !std::isfinite(L) || !(dt > 0.0) || !std::isfinite(dt))
        return efail(KG_EINVAL, "L and dt must be finite and > 0");
    for (int i = 0; i < count; i++) {
        if (Ns[i] != 64 && Ns[i] != 128) return efail(KG_ENOTSUP, "ensemble grids must be 64 or 128");
        if (!std::isfinite(A[i]) || !(s[i] > 0.0) || !std::isfinite(s[i])) return efail(KG_EINVAL, "bad A or s");
    }
    kg_options opt;
    kg_get_options(&opt);
    if (g_ens) {
        ens_destroy(g_ens);
        g_ens = nullptr;
    }
    Ens* e = new Ens();
    e->count = count;
    e->prec = opt.precision;
    e->pl = launcher_for(e->prec);
    e->L = L;
    e->dt = dt;
    e->lam = opt.nonlinearity;
    e->Ns.assign(Ns, Ns + count);
    const char* miss = std::getenv("KG_TEST_ENS_MISSING_CTA");   // test hook: force a wait to run out
    if (miss && std::atoi(miss) == 1) {
        e->missing = 1;
        e->spin_limit = 1ll << 16;
    }
    int rc = KG_OK;
#define KG_ETRY(x)          \
    do {                    \
        rc = (x);           \
        if (rc) {           \
            ens_destroy(e); \
            return rc;      \
        }                   \
    } while (0)
    {
        cudaError_t r = cudaStreamCreateWithFlags(&e->stream, cudaStreamNonBlocking);
        if (r != cudaSuccess) KG_ETRY(efail(KG_ECUDA, "cudaStreamCreate"));
        if (cudaEventCreate(&e->ev0) != cudaSuccess || cudaEventCreate(&e->ev1) != cudaSuccess)
            KG_ETRY(efail(KG_ECUDA, "cudaEventCreate"));
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&e->nsm, cudaDevAttrMultiProcessorCount, dev);
    }
    auto alloc = [e](void** p, size_t b, const char* w) { return ealloc(e, p, b, w); };
    int nmax = 0;
    for (int i = 0; i < count; i++) {
        const int t = Ns[i] == 64 ? 0 : 1;
        nmax = std::max(nmax, Ns[i]);
        if (!e->have[t]) {
            KG_ETRY(make_tables(Ns[i], e->prec, L, dt, alloc, &e->tab[t]));
            e->have[t] = true;
        }
    }
    const size_t spec_max = spec_slots(nmax, false);
    KG_ETRY(ealloc(e, (void**)&e->tmp, sizeof(double2) * spec_max, "ensemble spectral scratch"));
    KG_ETRY(ealloc(e, (void**)&e->tmp2, sizeof(double2) * spec_max, "ensemble spectral scratch"));
    static_assert(2 * kEnsMaxInst * sizeof(double) + kEnsMaxInst * sizeof(EnsAxis) <= (size_t)2 * 64 * 64 * 64 * 8,
                  "the set-up's 1D data fits the physical scratch");
    KG_ETRY(ealloc(e, (void**)&e->phys, sizeof(double) * std::max((size_t)nmax * nmax * nmax, (size_t)2 * 64 * 64 * 64),
                   "ensemble physical scratch"));
    // one allocation per array class, instances at 256-byte aligned offsets
    size_t off_s = 0, off_w = 0;
    std::vector<size_t> os(count), ow(count);
    for (int i = 0; i < count; i++) {
        const size_t ns = spec_slots(Ns[i], false);
        os[i] = off_s;
        ow[i] = off_w;
        off_s += (ns * sizeof(double2) + 255) & ~(size_t)255;
        off_w += (ns * e->pl->store_bytes + 255) & ~(size_t)255;
    }
    char *b0 = nullptr, *b1 = nullptr, *bw = nullptr, *bw2 = nullptr;
    KG_ETRY(ealloc(e, (void**)&b0, off_s, "ensemble S0"));
    KG_ETRY(ealloc(e, (void**)&b1, off_s, "ensemble S1"));
    KG_ETRY(ealloc(e, (void**)&bw, off_w, "ensemble W1"));
    KG_ETRY(ealloc(e, (void**)&bw2, off_w, "ensemble W2"));
    KG_ETRY(ealloc(e, (void**)&e->d_inst, sizeof(EnsInst) * count, "ensemble descriptors"));
    KG_ETRY(ealloc(e, (void**)&e->d_plan, sizeof(EnsPlan), "ensemble plan"));
    KG_ETRY(ealloc(e, (void**)&e->d_status, sizeof(int), "ensemble status"));
    KG_ETRY(ealloc(e, (void**)&e->d_order, sizeof(int) * count, "ensemble order"));
    KG_ETRY(ealloc(e, (void**)&e->d_feat, sizeof(double) * 4 * count, "ensemble features"));
    e->h_inst.resize(count);
    for (int i = 0; i < count; i++) {
        EnsInst& in = e->h_inst[i];
        std::memset(&in, 0, sizeof(in));
        in.S0 = (double2*)(b0 + os[i]);
        in.S1 = (double2*)(b1 + os[i]);
        in.W1 = (void*)(bw + ow[i]);
        in.W2 = (void*)(bw2 + ow[i]);
        in.N = Ns[i];
        in.blowup_level = -1;
    }
    // A, s and the 1D transforms travel through the physical scratch
    double* d_A = e->phys;
    double* d_s = d_A + kEnsMaxInst;
    EnsAxis* axis = reinterpret_cast<EnsAxis*>(d_s + kEnsMaxInst);
    if (cudaMemcpyAsync(e->d_inst, e->h_inst.data(), sizeof(EnsInst) * count, cudaMemcpyHostToDevice, e->stream) != cudaSuccess ||
        cudaMemcpyAsync(d_A, A, sizeof(double) * count, cudaMemcpyHostToDevice, e->stream) != cudaSuccess ||
        cudaMemcpyAsync(d_s, s, sizeof(double) * count, cudaMemcpyHostToDevice, e->stream) != cudaSuccess ||
        cudaMemsetAsync(e->d_status, 0, sizeof(int), e->stream) != cudaSuccess)
        KG_ETRY(efail(KG_ECUDA, "ensemble state upload"));
    k_ens_axis<<<count, 128, 0, e->stream>>>(e->d_inst, d_s, L, e->tab[0].tw64, e->tab[1].tw64, axis);
    if (cudaGetLastError() != cudaSuccess ||
        e->pl->ens_fill(e->d_inst, count, axis, d_A, e->lam, e->tab[0].coef, e->tab[1].coef, e->stream) != cudaSuccess)
        KG_ETRY(efail(KG_ECUDA, "ensemble set-up launch"));
    if (e->pl->store_bytes != sizeof(double2)) {
        // FP32 work arrays: the inverse z and y transforms of uh^0, as a step leaves them
        for (int i = 0; i < count; i++) {
            const EnsInst& in = e->h_inst[i];
            const Tables& tb = e->tab[in.N == 64 ? 0 : 1];
            if (e->pl->z_from_f64(in.N, in.S0, in.S1, nullptr, in.W2, tb.tw, e->pl->lg(in.N), e->stream) != cudaSuccess ||
                e->pl->yi(in.N, in.W2, in.W1, tb.tw, e->pl->lg(in.N), FinArgs{}, e->stream) != cudaSuccess)
                KG_ETRY(efail(KG_ECUDA, "ensemble set-up transforms"));
        }
    }
    // (the layout is the same for both grids)
    k_shells<<<count, 256, 0, e->stream>>>(e->d_inst, e->pl->lg(64), L, e->d_feat);
    if (cudaGetLastError() != cudaSuccess) KG_ETRY(efail(KG_ECUDA, "shells launch"));
    if (cudaStreamSynchronize(e->stream) != cudaSuccess) KG_ETRY(efail(KG_ECUDA, "ensemble init"));
    e->threshold = -1.0;
    {
        int n64, n128;
        count_sizes(e->Ns, &n64, &n128);
        Tuned t;
        const bool use = (g_tuned.valid && g_tuned.prec == e->prec && g_tuned.n64 == n64 && g_tuned.n128 == n128 &&
                          (t = g_tuned, true)) ||
                         cache_lookup(e->prec, n64, n128, &t);
        // untuned: as many CTAs as fit, fewer where a pass has few units for each; half-width
        // tiles for FP32 (256 x 64^3: 0.79 ms per step against 0.85; 16-byte precisions no gain).
        // ms per step double-float with 2, 3, 4 CTAs per SM: 8 x 64^3 (640 units) 0.075, 0.074,
        // 0.083; 128^3 (576) 0.088, 0.112, 0.109; 3 + 1 (816) 0.127, 0.127, 0.154; 12 x 64^3 (960)
        // 0.110, 0.092, 0.094; 2 x 128^3 (1152) 0.152, 0.140, 0.133; 24 x 64^3 0.195, 0.176, 0.163
        const int sched = e->pl->store_bytes == 8 ? 1 : 0;
        const int maxb = e->pl->ens_blocks_per_sm(sched), units = pass_units(n64, n128);
        const int bps = std::min(maxb, units < 5 * e->nsm ? 2 : units < 6 * e->nsm ? 3 : maxb);
        KG_ETRY(set_shape(e, use ? t.sched : sched, use ? t.bps : bps, use ? t.order : 1));
    }
#undef KG_ETRY
    g_ens = e;
    return KG_OK;
}

int kg_ens_run(int max_steps, double threshold, long long* steps_done, double* ms) {
    Ens* e = g_ens;
    if (!e) return efail(KG_ESTATE, "kg_ens_run before kg_ens_init");
    if (max_steps < 0 || !std::isfinite(threshold)) return efail(KG_EINVAL, "bad arguments");
    e->threshold = threshold;
    long long done = 0;
    KG_ECK(cudaEventRecord(e->ev0, e->stream));
    while (done < max_steps) {
        const int n = (int)std::min<long long>(max_steps - done, kLaunchSteps);
        int rl = launch_steps(e, n);
        if (rl) return rl;
        done += n;
        {
            // stop early once every instance has blown up
            KG_ECK(cudaMemcpyAsync(e->h_inst.data(), e->d_inst, sizeof(EnsInst) * e->count, cudaMemcpyDeviceToHost,
                                   e->stream));
            KG_ECK(cudaStreamSynchronize(e->stream));
            int rc = check_status(e);
            if (rc) return rc;
            bool any = false;
            for (const EnsInst& in : e->h_inst) any = any || !in.frozen;
            if (!any) break;
        }
    }
    KG_ECK(cudaEventRecord(e->ev1, e->stream));
    KG_ECK(cudaEventSynchronize(e->ev1));
    int rc = check_status(e);
    if (rc) return rc;
    float t = 0.f;
    KG_ECK(cudaEventElapsedTime(&t, e->ev0, e->ev1));
    if (steps_done) *steps_done = done;
    if (ms) *ms = t;
    return KG_OK;
}

int kg_ens_results(int* frozen, long long* blowup_level, long long* level, double* maxabs) {
    Ens* e = g_ens;
    if (!e) return efail(KG_ESTATE, "kg_ens_results before kg_ens_init");
    KG_ECK(cudaStreamSynchronize(e->stream));
    KG_ECK(cudaMemcpy(e->h_inst.data(), e->d_inst, sizeof(EnsInst) * e->count, cudaMemcpyDeviceToHost));
    for (int i = 0; i < e->count; i++) {
        const EnsInst& in = e->h_inst[i];
        if (frozen) frozen[i] = in.frozen;
        if (blowup_level) blowup_level[i] = in.blowup_level;
        if (level) level[i] = in.level;
        if (maxabs) maxabs[i] = in.maxabs;
    }
    return KG_OK;
}

int kg_ens_features(double* shells) {
    Ens* e = g_ens;
    if (!e) return efail(KG_ESTATE, "kg_ens_features before kg_ens_init");
    if (!shells) return efail(KG_EINVAL, "NULL");
    KG_ECK(cudaStreamSynchronize(e->stream));
    KG_ECK(cudaMemcpy(shells, e->d_feat, sizeof(double) * 4 * e->count, cudaMemcpyDeviceToHost));
    return KG_OK;
}

int kg_ens_fetch(int i, double* u) {
    Ens* e = g_ens;
    if (!e) return efail(KG_ESTATE, "kg_ens_fetch before kg_ens_init");
    if (i < 0 || i >= e->count || !u) return efail(KG_EINVAL, "bad instance index or NULL");
    KG_ECK(cudaStreamSynchronize(e->stream));
    EnsInst in;
    KG_ECK(cudaMemcpy(&in, e->d_inst + i, sizeof(EnsInst), cudaMemcpyDeviceToHost));
    const int N = in.N;
    const Tables& tb = e->tab[N == 64 ? 0 : 1];
    const double2* cur = in.phase ? in.S1 : in.S0;
    KG_ECK(kLaunchF64.z_from_f64(N, cur, cur, nullptr, e->tmp2, tb.tw64, e->pl->lg(N), e->stream));
    KG_ECK(kLaunchF64.yi(N, e->tmp2, e->tmp, tb.tw64, e->pl->lg(N), FinArgs{}, e->stream));
    KG_ECK(launch_x_inverse(N, e->tmp, e->phys, tb.tw64, 1.0 / ((double)N * N * N), nullptr, e->stream));
    KG_ECK(cudaMemcpyAsync(u, e->phys, sizeof(double) * (size_t)N * N * N, cudaMemcpyDeviceToHost, e->stream));
    KG_ECK(cudaStreamSynchronize(e->stream));
    return KG_OK;
}

int kg_ens_tune(int steps, int* blocks_per_sm, int* order) {
    Ens* e = g_ens;
    if (!e) return efail(KG_ESTATE, "kg_ens_tune before kg_ens_init");
    if (steps < 1) return efail(KG_EINVAL, "steps < 1");
    // the candidates advance the ensemble itself: tune on a throw-away ensemble and
    // initialise the measured one afterwards (the choice is kept for it).  Candidates:
    // every schedule (tile width x stage order) x unit order x resident CTAs per SM
    float best = 1e30f;
    int bs = 0, bb = 1, bo = 0;
    for (int sc = 0; sc < kEnsSchedules; sc++) {
        const int maxb = e->pl->ens_blocks_per_sm(sc);
        for (int o = 0; o < 2; o++) {
            for (int b = 1; b <= maxb; b++) {
                int rc = set_shape(e, sc, b, o);
                if (rc) return rc;
                rc = launch_steps(e, 1);   // warm-up
                if (rc) return rc;
                KG_ECK(cudaEventRecord(e->ev0, e->stream));
                rc = launch_steps(e, steps);
                if (rc) return rc;
                KG_ECK(cudaEventRecord(e->ev1, e->stream));
                KG_ECK(cudaEventSynchronize(e->ev1));
                int rs = check_status(e);
                if (rs) return rs;
                float t = 0.f;
                KG_ECK(cudaEventElapsedTime(&t, e->ev0, e->ev1));
                if (t < best) {
                    best = t;
                    bs = sc;
                    bb = b;
                    bo = o;
                }
            }
        }
    }
    int rc = set_shape(e, bs, bb, bo);
    if (rc) return rc;
    g_tuned.valid = true;
    g_tuned.prec = e->prec;
    count_sizes(e->Ns, &g_tuned.n64, &g_tuned.n128);
    g_tuned.sched = bs;
    g_tuned.bps = bb;
    g_tuned.order = bo;
    rc = cache_store(g_tuned, best / steps);
    if (rc) return rc;
    if (blocks_per_sm) *blocks_per_sm = bb;
    if (order) *order = bo;
    return KG_OK;
}

int kg_ens_schedule(int* sched, int* blocks_per_sm, int* order) {
    Ens* e = g_ens;
    if (!e) return efail(KG_ESTATE, "kg_ens_schedule before kg_ens_init");
    if (sched) *sched = e->sched;
    if (blocks_per_sm) *blocks_per_sm = e->bps;
    if (order) *order = e->order;
    return KG_OK;
}

int kg_ens_set_schedule(int sched, int blocks_per_sm, int order) {
    Ens* e = g_ens;
    if (!e) return efail(KG_ESTATE, "kg_ens_set_schedule before kg_ens_init");
    if (sched < 0 || sched >= kEnsSchedules || blocks_per_sm < 1 || (order != 0 && order != 1))
        return efail(KG_EINVAL, "kg_ens_set_schedule: sched in [0, 4), blocks_per_sm >= 1, order 0 or 1");
    KG_ECK(cudaStreamSynchronize(e->stream));
    return set_shape(e, sched, blocks_per_sm, order);
}

int kg_ens_set_tune_cache(const char* path) {
    g_cache_path = path ? path : "";
    return KG_OK;
}

int kg_gaussian_features(int count, int N, double L, const double* A, const double* s, double* shells) {
    if (count < 1 || N < 10 || (N & 1) || !(L > 0.0) || !A || !s || !shells) return efail(KG_EINVAL, "bad arguments");
    double *dA = nullptr, *dS = nullptr, *dO = nullptr;
    if (cudaMalloc((void**)&dA, sizeof(double) * count) != cudaSuccess ||
        cudaMalloc((void**)&dS, sizeof(double) * count) != cudaSuccess ||
        cudaMalloc((void**)&dO, sizeof(double) * 4 * (size_t)count) != cudaSuccess) {
        cudaFree(dA);
        cudaFree(dS);
        cudaGetLastError();
        return efail(KG_ENOMEM, "feature buffers");
    }
    cudaError_t e = cudaMemcpy(dA, A, sizeof(double) * count, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dS, s, sizeof(double) * count, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_gauss_shells<<<(count + 127) / 128, 128>>>(count, N, L, dA, dS, dO);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(shells, dO, sizeof(double) * 4 * (size_t)count, cudaMemcpyDeviceToHost);
    cudaFree(dA);
    cudaFree(dS);
    cudaFree(dO);
    if (e != cudaSuccess) return efail(KG_ECUDA, std::string("gaussian features: ") + cudaGetErrorString(e));
    return KG_OK;
}

int kg_ens_finalize(void) {
    if (g_ens) {
        ens_destroy(g_ens);
        g_ens = nullptr;
    }
    return KG_OK;
}

}  // extern "C"

namespace kg {
// the autotuner's cache file for kg_get_options (NULL when there is none)
const char* ens_tune_cache() { return g_cache_path.empty() ? nullptr : g_cache_path.c_str(); }
}  // namespace kg
