// C-ABI entry points (include/hf.h): argument checks, device memory, and the
// order of the setup and Fock-build kernels on the context's stream.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "eri_common.cuh"
#include "hf_internal.h"
#include "setup.cuh"

namespace hf {

static thread_local std::string g_err;

void set_error(int code, const std::string& msg)
{
    (void)code;
    g_err = msg;
}

int cuda_status(cudaError_t e, const char* what)
{
    g_err = std::string(what) + ": " + cudaGetErrorString(e);
    cudaGetLastError();
    return HF_E_CUDA;
}

int DevBuf::alloc(size_t n)
{
    release();
    owned = true;
    if (n == 0) n = 16;
    cudaError_t e = cudaMalloc(&p, n);
    if (e != cudaSuccess) {
        p = nullptr;
        cudaGetLastError();
        g_err = "device allocation of " + std::to_string(n) + " bytes failed";
        return HF_E_NOMEM;
    }
    bytes = n;
    return HF_OK;
}

void DevBuf::release()
{
    if (p && owned) cudaFree(p);
    p = nullptr;
    bytes = 0;
    owned = true;
}

void add_exponents(std::vector<double>& exps, const hf_basis& b)
{
    long long n = 0;
    for (int s = 0; s < b.n_shells; s++) n += b.nprim[s];
    exps.insert(exps.end(), b.exps, b.exps + n);
    std::sort(exps.begin(), exps.end());
    exps.erase(std::unique(exps.begin(), exps.end()), exps.end());
}

int exponent_table(hf_ctx* ctx, std::vector<double> exps, std::shared_ptr<const ExponentTable>& out)
{
    std::lock_guard<std::mutex> lock(ctx->tables_lock);
    auto& all = ctx->tables;
    all.erase(std::remove_if(all.begin(), all.end(), [](const auto& w) { return w.expired(); }), all.end());
    for (const auto& w : all) {
        out = w.lock();
        if (out && out->exps == exps) return HF_OK;
    }
    auto t = std::make_shared<ExponentTable>();
    t->exps = std::move(exps);
    const int rc = t->build(ctx->stream);
    out = rc == HF_OK ? t : nullptr;
    if (rc == HF_OK) all.push_back(t);
    return rc;
}

int ExponentTable::build(cudaStream_t s)
{
    const long long n = (long long)exps.size(), nt = n * (n + 1) / 2;
    if (nt > kHermMaxTypes) return HF_OK;
    std::vector<double> ps;
    for (int i = 0; i < n; i++)
        for (int j = 0; j <= i; j++) ps.push_back(exps[i] + exps[j]);  // type i (i + 1) / 2 + j
    int rc = psum.alloc(sizeof(double) * nt);
    if (rc == HF_OK) rc = tab.alloc(sizeof(double2) * nt * nt);
    if (rc != HF_OK) return rc;
    HF_CUDA(cudaMemcpyAsync(psum.p, ps.data(), sizeof(double) * nt, cudaMemcpyHostToDevice, s));
    HF_CUDA(cudaStreamSynchronize(s));  // ps goes out of scope
    ntype = (int)nt;
    return launch_exponent_table(ntype, psum.as<double>(), tab.as<double2>(), s) == 0
               ? HF_OK : cuda_status(cudaGetLastError(), "exponent table");
}

namespace {

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

int fail(int code, const std::string& msg)
{
    g_err = msg;
    return code;
}

#define TRY(x)                       \
    do {                             \
        int rc_ = (x);               \
        if (rc_ != HF_OK) return rc_; \
    } while (0)

#define KCHK(x)                                                                  \
    do {                                                                         \
        if ((x) != 0) return cuda_status(cudaGetLastError(), "kernel launch " #x); \
    } while (0)

size_t next_pow2(size_t n)
{
    size_t p = 1;
    while (p < n) p <<= 1;
    return p;
}

int class_index(int X, int Y)
{
    for (int c = 0; c < kNumClasses; c++)
        if (kEriClasses[c].X == X && kEriClasses[c].Y == Y) return c;
    return -1;
}

}  // namespace

}  // namespace hf

using namespace hf;

extern "C" {

const char* hf_strerror(int status)
{
    switch (status) {
        case HF_OK: return "success";
        case HF_E_INVALID: return "invalid argument";
        case HF_E_UNSUPPORTED: return "unsupported input or device";
        case HF_E_NOMEM: return "out of memory";
        case HF_E_CUDA: return "CUDA runtime error";
        case HF_E_TIMEOUT: return "device wait timed out";
        case HF_E_NOCONV: return "SCF did not converge";
        default: return "unknown status";
    }
}

const char* hf_last_error(void) { return g_err.c_str(); }

static void ctx_release(hf_ctx* c)
{
    DeviceGuard g(c->device);
    for (auto& ev : c->ev)
        if (ev) cudaEventDestroy(ev);
    for (auto& e : c->join)
        if (e) cudaEventDestroy(e);
    for (auto& s : c->side)
        if (s) cudaStreamDestroy(s);
    if (c->fast) cudaStreamDestroy(c->fast);
    if (c->fork) cudaEventDestroy(c->fork);
    delete c;
}

int hf_create(hf_ctx** out, int device, void* cuda_stream)
{
    if (!out) return fail(HF_E_INVALID, "hf_create: ctx pointer is NULL");
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
        cudaGetLastError();
        return fail(HF_E_UNSUPPORTED, "hf_create: no CUDA device");
    }
    if (device < 0 || device >= ndev) return fail(HF_E_INVALID, "hf_create: device index out of range");
    cudaDeviceProp prop;
    HF_CUDA(cudaGetDeviceProperties(&prop, device));
    if (prop.major != 10 || prop.minor != 3)
        return fail(HF_E_UNSUPPORTED, "hf_create: library is built for sm_103a (GB300); device is sm_" +
                                          std::to_string(prop.major) + std::to_string(prop.minor));
    DeviceGuard g(device);
    hf_ctx* c = new hf_ctx();
    c->device = device;
    c->stream = (cudaStream_t)cuda_stream;
    c->num_sms = prop.multiProcessorCount;
    int rc = c->boys64.alloc(sizeof(double) * kBoysRows64 * kBoysStride64);
    if (rc == HF_OK) rc = c->boys32.alloc(sizeof(float) * kBoysRows32 * kBoysStride32);
    if (rc == HF_OK && build_boys_tables(c->boys64.as<double>(), c->boys32.as<float>(), c->stream) != 0)
        rc = cuda_status(cudaGetLastError(), "boys table kernel");
    if (rc == HF_OK) {
        cudaError_t e = cudaStreamSynchronize(c->stream);
        if (e != cudaSuccess) rc = cuda_status(e, "hf_create sync");
    }
    if (rc == HF_OK) {
        // Reserve per-thread local memory for the largest ERI kernel once, so that launches of the
        // spilling high-angular-momentum kernels do not grow and shrink the reservation each time.
        size_t need = 0;
        for (int ci = 0; ci < kNumClasses; ci++) {
            need = std::max(need, kEriClasses[ci].local_bytes());
            if (kEriClasses[ci].local_bytes_rys) need = std::max(need, kEriClasses[ci].local_bytes_rys());
            need = std::max(need, kEriClasses[ci].local_bytes_h());
            if (kEriClasses[ci].prepare() != 0) rc = cuda_status(cudaGetLastError(), "hf_create: shared memory limit");
        }
        size_t cur = 0;
        if (cudaDeviceGetLimit(&cur, cudaLimitStackSize) == cudaSuccess && need > cur)
            if (cudaDeviceSetLimit(cudaLimitStackSize, need) != cudaSuccess)
                rc = cuda_status(cudaGetLastError(), "hf_create: local memory reservation");
        cudaGetLastError();
    }
    // the allocation-free build's fixed scratch: looking its address up loads its module now, so that
    // the driver reserves that memory here and not inside an hf_fock_build_noalloc call
    if (rc == HF_OK) rc = noalloc_scratch_address(&c->noalloc_scratch);
    if (rc == HF_OK) {
        for (auto& ev : c->ev) {
            if (cudaEventCreate(&ev) != cudaSuccess) {
                rc = cuda_status(cudaGetLastError(), "cudaEventCreate");
                break;
            }
        }
        int least = 0, greatest = 0;
        cudaDeviceGetStreamPriorityRange(&least, &greatest);
        for (int i = 0; i <= kSideStreams && rc == HF_OK; i++)
            if (cudaStreamCreateWithPriority(i < kSideStreams ? &c->side[i] : &c->fast, cudaStreamNonBlocking,
                                             i < kSideStreams ? least : greatest) != cudaSuccess ||
                cudaEventCreateWithFlags(&c->join[i], cudaEventDisableTiming) != cudaSuccess)
                rc = cuda_status(cudaGetLastError(), "hf_create: side stream");
        if (rc == HF_OK && cudaEventCreateWithFlags(&c->fork, cudaEventDisableTiming) != cudaSuccess)
            rc = cuda_status(cudaGetLastError(), "cudaEventCreate");
    }
    if (rc != HF_OK) {
        ctx_release(c);
        return rc;
    }
    *out = c;
    return HF_OK;
}

void hf_destroy(hf_ctx* c)
{
    if (!c) return;
    if (c->n_systems > 0) {  // released together with its last system
        c->destroy_pending = true;
        return;
    }
    ctx_release(c);
}

}  // extern "C"

// Carves 256-byte-aligned views out of one allocation.
struct Arena {
    size_t used = 0;
    std::vector<std::pair<DevBuf*, size_t>> items;
    void add(DevBuf& b, size_t bytes)
    {
        items.push_back({&b, used});
        b.bytes = bytes;
        used += (bytes + 255) & ~(size_t)255;
    }
    int commit(DevBuf& owner)
    {
        TRY(owner.alloc(used ? used : 256));
        for (auto& it : items) {
            const size_t n = it.first->bytes;
            it.first->view((char*)owner.p + it.second, n);
        }
        return HF_OK;
    }
};

// The context's side streams between an event recorded on its stream and one it waits for; the destructor joins
// what an early return left running, which still uses the caller's buffers.
struct SideStreams {
    hf_ctx* ctx;
    bool open = false;
    explicit SideStreams(hf_ctx* c) : ctx(c) {}
    int fork()
    {
        HF_CUDA(cudaEventRecord(ctx->fork, ctx->stream));
        open = true;
        for (auto& s : ctx->side) HF_CUDA(cudaStreamWaitEvent(s, ctx->fork, 0));
        HF_CUDA(cudaStreamWaitEvent(ctx->fast, ctx->fork, 0));
        return HF_OK;
    }
    int join()
    {
        if (!open) return HF_OK;
        open = false;
        cudaError_t err = cudaSuccess;
        for (int i = 0; i <= kSideStreams; i++) {
            const cudaError_t e1 = cudaEventRecord(ctx->join[i], i < kSideStreams ? ctx->side[i] : ctx->fast);
            const cudaError_t e2 = cudaStreamWaitEvent(ctx->stream, ctx->join[i], 0);
            if (err == cudaSuccess) err = e1 != cudaSuccess ? e1 : e2;
        }
        return err == cudaSuccess ? HF_OK : cuda_status(err, "joining the side streams");
    }
    ~SideStreams() { join(); }
};

static int system_setup(hf_system* S, const hf_geometry* geom, const hf_basis* basis)
{
    hf_ctx* ctx = S->ctx;
    cudaStream_t st = ctx->stream;
    hf_system& X = *S;
    const int na = geom->n_atoms, ns = basis->n_shells;
    // host bookkeeping of the basis layout (offsets only)
    std::vector<int> bf0(ns), prim0(ns);
    int nbf = 0, npr = 0, maxnp = 0;
    for (int s = 0; s < ns; s++) {
        bf0[s] = nbf;
        prim0[s] = npr;
        nbf += (basis->l[s] + 1) * (basis->l[s] + 2) / 2;
        npr += basis->nprim[s];
        maxnp = std::max(maxnp, (int)basis->nprim[s]);
    }
    std::vector<double> Zd(na);
    int nel = 0;
    for (int a = 0; a < na; a++) {
        Zd[a] = geom->Z[a];
        nel += geom->Z[a];
    }
    S->Z_h.assign(geom->Z, geom->Z + na);
    S->atom_bf0_h.assign(na, -1);
    S->atom_nbf_h.assign(na, 0);
    {
        int last = -1;
        for (int s = 0; s < ns; s++) {
            const int a = basis->atom[s];
            if (S->atom_bf0_h[a] < 0) S->atom_bf0_h[a] = bf0[s];
            else if (last != a) S->atom_nbf_h[a] = -1000000;  // shells of this atom are not contiguous
            S->atom_nbf_h[a] += (basis->l[s] + 1) * (basis->l[s] + 2) / 2;
            last = a;
        }
        for (int a = 0; a < na; a++)
            if (S->atom_nbf_h[a] < 0) S->atom_bf0_h[a] = -1;
    }
    S->n_atoms = na;
    S->n_shells = ns;
    S->n_bf = nbf;
    S->n_electrons = nel;
    X.maxpp = maxnp * maxnp;
    const long long npairs = (long long)ns * (ns + 1) / 2;
    if (npairs * (long long)X.maxpp >= (1ll << 31)) return fail(HF_E_UNSUPPORTED, "too many primitive pairs");
    S->n_pairs_all = (int)npairs;
    const size_t NN = (size_t)nbf * nbf;

    // exponent table and each primitive's place in it
    if (!S->etab) {
        std::vector<double> exps;
        add_exponents(exps, *basis);
        TRY(exponent_table(ctx, std::move(exps), S->etab));
    }
    const ExponentTable* const table = S->etab.get();
    std::vector<int> utype(npr);
    for (int k = 0; k < npr; k++)
        utype[k] = (int)(std::lower_bound(table->exps.begin(), table->exps.end(), basis->exps[k]) - table->exps.begin());

    // ---------------------------------------------- inputs, matrices, pairs
    DevBuf utype_in;
    DevBuf coef_in;
    Arena a1;
    a1.add(S->sh_l, sizeof(int) * ns);
    a1.add(S->sh_atom, sizeof(int) * ns);
    a1.add(S->sh_bf0, sizeof(int) * ns);
    a1.add(S->sh_nprim, sizeof(int) * ns);
    a1.add(S->sh_prim0, sizeof(int) * ns);
    a1.add(S->sh_exp, sizeof(double) * npr);
    a1.add(coef_in, sizeof(double) * npr);
    a1.add(S->atom_xyz, sizeof(double) * 3 * na);
    a1.add(S->atom_Z, sizeof(double) * na);
    a1.add(S->sh_coef, sizeof(double) * npr);
    a1.add(S->comp_norm, sizeof(double) * nbf);
    a1.add(S->Ebuf, sizeof(double) * 320);
    a1.add(S->pairs, sizeof(PairHdr) * npairs);
    a1.add(S->prims64, sizeof(PrimPair<double>) * npairs * X.maxpp);
    a1.add(S->prims32, sizeof(PrimPair<float>) * npairs * X.maxpp);
    a1.add(utype_in, sizeof(int) * npr);
    a1.add(S->hrec, sizeof(HermPair) * npairs * X.maxpp);
    a1.add(S->hB, sizeof(float) * npairs * X.maxpp);
    a1.add(S->pair_class, sizeof(int) * npairs);
    a1.add(X.counts, sizeof(unsigned long long) * 16);
    a1.add(X.Qall, sizeof(double) * npairs);
    a1.add(X.Bprim, sizeof(double) * npairs * X.maxpp);
    TRY(a1.commit(X.arena_in));
    Arena a2;
    a2.add(S->S, NN * sizeof(double));
    a2.add(S->H, NN * sizeof(double));
    a2.add(S->P64, NN * sizeof(double));
    if (S->th.fp32_cutoff > 0.0) a2.add(S->P32, NN * sizeof(float));
    a2.add(S->Jt, NN * sizeof(double));
    a2.add(S->Kt, NN * sizeof(double));
    a2.add(S->F, NN * sizeof(double));
    a2.add(X.staging_P, NN * sizeof(double));
    a2.add(X.staging_out, 2 * NN * sizeof(double));
    a2.add(X.bad, sizeof(int));
    a2.add(X.prim_count, sizeof(unsigned long long) * 2 * kNumClasses);
    TRY(a2.commit(X.arena_mat));
    HF_CUDA(cudaMemcpyAsync(S->sh_l.p, basis->l, sizeof(int) * ns, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemcpyAsync(S->sh_atom.p, basis->atom, sizeof(int) * ns, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemcpyAsync(S->sh_bf0.p, bf0.data(), sizeof(int) * ns, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemcpyAsync(S->sh_nprim.p, basis->nprim, sizeof(int) * ns, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemcpyAsync(S->sh_prim0.p, prim0.data(), sizeof(int) * ns, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemcpyAsync(S->sh_exp.p, basis->exps, sizeof(double) * npr, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemcpyAsync(coef_in.p, basis->coefs, sizeof(double) * npr, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemcpyAsync(S->atom_xyz.p, geom->xyz, sizeof(double) * 3 * na, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemcpyAsync(S->atom_Z.p, Zd.data(), sizeof(double) * na, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemcpyAsync(utype_in.p, utype.data(), sizeof(int) * npr, cudaMemcpyHostToDevice, st));
    HF_CUDA(cudaMemsetAsync(S->hB.p, 0, sizeof(float) * npairs * X.maxpp, st));
    S->herm.rec = S->hrec.as<HermPair>();
    S->herm.B = S->hB.as<float>();
    S->herm = table->view(S->herm);
    KCHK(launch_shell_coef(ns, S->sh_l.as<int>(), S->sh_nprim.as<int>(), S->sh_prim0.as<int>(), S->sh_exp.as<double>(),
                           coef_in.as<double>(), S->sh_coef.as<double>(), st));
    KCHK(launch_comp_norm(ns, S->sh_l.as<int>(), S->sh_bf0.as<int>(), S->comp_norm.as<double>(), st));
    KCHK(launch_nuclear_repulsion(na, S->atom_xyz.as<double>(), S->atom_Z.as<double>(), S->Ebuf.as<double>() + 300,
                                  st));
    KCHK(launch_build_pairs(npairs, X.maxpp, S->sh_l.as<int>(), S->sh_atom.as<int>(), S->sh_bf0.as<int>(),
                            S->sh_nprim.as<int>(), S->sh_prim0.as<int>(), S->sh_exp.as<double>(),
                            S->sh_coef.as<double>(), S->atom_xyz.as<double>(), S->pairs.as<PairHdr>(),
                            S->prims64.p, S->prims32.p, S->hrec.as<HermPair>(), utype_in.as<int>(),
                            S->pair_class.as<int>(), st));
    unsigned long long* cnt_dev = X.counts.as<unsigned long long>();  // [0..5] class counts, [8..15] cursors
    HF_CUDA(cudaMemsetAsync(cnt_dev, 0, sizeof(unsigned long long) * 16, st));
    KCHK(launch_class_count(npairs, S->pair_class.as<int>(), cnt_dev, st));
    unsigned long long cnt_all[kNumPairClasses];
    HF_CUDA(cudaMemcpyAsync(cnt_all, cnt_dev, sizeof(cnt_all), cudaMemcpyDeviceToHost, st));
    HF_CUDA(cudaStreamSynchronize(st));  // host sync: class sizes

    // ------------------------------------------------------ schedule arena
    size_t npad[kNumPairClasses], seg[kNumPairClasses + 1], base_all[kNumPairClasses + 1];
    seg[0] = base_all[0] = 0;
    for (int c = 0; c < kNumPairClasses; c++) {
        npad[c] = cnt_all[c] ? next_pow2(cnt_all[c]) : 0;
        seg[c + 1] = seg[c] + npad[c];
        base_all[c + 1] = base_all[c] + cnt_all[c];
    }
    DevBuf ids_all, key, val, rb;
    DevBuf c64[kNumClasses], c32[kNumClasses];
    Arena a3;
    a3.add(ids_all, sizeof(int) * (npairs ? npairs : 1));
    a3.add(key, sizeof(double) * (seg[kNumPairClasses] ? seg[kNumPairClasses] : 1));
    a3.add(val, sizeof(int) * (seg[kNumPairClasses] ? seg[kNumPairClasses] : 1));
    a3.add(rb, 512);  // readback block: unsigned nsig[8] | long long totals[2*21] | double E_nn
    for (int ci = 0; ci < kNumClasses; ci++) {
        const size_t cap = cnt_all[kEriClasses[ci].X];
        auto& pl = S->plan[ci];
        a3.add(c64[ci], sizeof(long long) * (cap ? cap : 1));
        a3.add(c32[ci], sizeof(long long) * (cap ? cap : 1));
        a3.add(pl.kstart32, sizeof(int) * (cap ? cap : 1));
        a3.add(pl.offsets64, sizeof(long long) * (cap + 1));
        a3.add(pl.offsets32, sizeof(long long) * (cap + 1));
    }
    TRY(a3.commit(X.arena_sched));
    unsigned* nsig_dev = rb.as<unsigned>();
    long long* totals_dev = (long long*)(rb.as<char>() + 32);
    double* enn_dev = (double*)(rb.as<char>() + 32 + 8 * 2 * kNumClasses);
    HF_CUDA(cudaMemsetAsync(rb.p, 0, 512, st));

    // --------------------------------------------------- Schwarz bounds
    HF_CUDA(cudaMemsetAsync(X.Qall.p, 0, sizeof(double) * npairs, st));
    HF_CUDA(cudaMemsetAsync(X.Bprim.p, 0, sizeof(double) * npairs * X.maxpp, st));
    for (int c = 0; c < kNumPairClasses; c++)
        if (cnt_all[c])
            KCHK(launch_class_scatter_all(npairs, S->pair_class.as<int>(), c, (unsigned*)(cnt_dev + 8 + c),
                                          ids_all.as<int>() + base_all[c], st));
    // bounds and one-electron blocks of the classes run concurrently: each lasts as long as its longest pair
    {
        SideStreams side(ctx);
        TRY(side.fork());
        for (int c = 0; c < kNumPairClasses; c++) {
            if (!cnt_all[c]) continue;
            int* ids = ids_all.as<int>() + base_all[c];
            SchwarzArgs sa;
            sa.pairs = S->pairs.as<PairHdr>();
            sa.herm = S->herm;
            sa.ids = ids;
            sa.n = (int)cnt_all[c];
            sa.Q = X.Qall.as<double>();
            sa.boys64 = ctx->boys64.as<double>();
            sa.Bprim = X.Bprim.as<double>();
            sa.items = X.maxpp + 1;
            kEriClasses[class_index(c, c)].launch_schwarz(sa, kEriThreads, ctx->side[c]);
            HF_CUDA(cudaGetLastError());
            OneEArgs oa{S->pairs.as<PairHdr>(), ids, (int)cnt_all[c], na, nbf, S->sh_nprim.as<int>(),
                        S->sh_prim0.as<int>(), S->sh_exp.as<double>(), S->sh_coef.as<double>(),
                        S->atom_xyz.as<double>(), S->atom_Z.as<double>(), S->comp_norm.as<double>(),
                        ctx->boys64.as<double>(), S->herm, S->S.as<double>(), S->H.as<double>()};
            KCHK(launch_one_electron_class(c, oa, ctx->side[(c + 3) % kSideStreams]));
        }
        TRY(side.join());
    }
    KCHK(launch_sort_prims(npairs, S->pairs.as<PairHdr>(), X.Bprim.as<double>(), S->prims64.p, S->prims32.p,
                           S->hrec.as<HermPair>(), S->hB.as<float>(), st));
    unsigned long long* qbits_dev = cnt_dev + 7;
    HF_CUDA(cudaMemsetAsync(qbits_dev, 0, sizeof(unsigned long long), st));
    KCHK(launch_copy_q(npairs, X.Qall.as<double>(), S->pairs.as<PairHdr>(), qbits_dev, st));

    // ------------------------------------- significant pairs, sorted by Q
    const double tau = S->th.schwarz_tau;
    KCHK(launch_sig_scatter(npairs, (long long)seg[kNumPairClasses], S->pair_class.as<int>(), X.Qall.as<double>(),
                            qbits_dev, tau, seg, nsig_dev, key.as<double>(), val.as<int>(), st));
    SideStreams sorts(ctx);
    TRY(sorts.fork());
    for (int c = 0; c < kNumPairClasses; c++) {
        if (!npad[c]) continue;
        KCHK(bitonic_sort_desc(key.as<double>() + seg[c], val.as<int>() + seg[c], (int)npad[c], (int)npad[c],
                               ctx->side[c]));
        S->class_ids[c].view(val.as<int>() + seg[c], sizeof(int) * npad[c]);
        X.class_q[c].view(key.as<double>() + seg[c], sizeof(double) * npad[c]);
    }

    TRY(sorts.join());

    // ------------------------------------------------- quartet schedule
    S->quartets_total = 0;
    QuartetSchedule qs{};
    qs.tau = tau;
    qs.cutoff = S->th.fp32_cutoff;
    qs.totals = totals_dev;
    for (int ci = 0; ci < kNumClasses; ci++) {
        const int Xc = kEriClasses[ci].X, Yc = kEriClasses[ci].Y;
        auto& pl = S->plan[ci];
        pl.n_unscreened = (Xc == Yc) ? (long long)cnt_all[Xc] * (cnt_all[Xc] + 1) / 2
                                     : (long long)cnt_all[Xc] * (long long)cnt_all[Yc];
        S->quartets_total += pl.n_unscreened;
        if (!cnt_all[Xc] || !cnt_all[Yc]) continue;
        qs.c[ci] = {(int)cnt_all[Xc], Xc == Yc, nsig_dev + Xc, nsig_dev + Yc, X.class_q[Xc].as<double>(),
                    X.class_q[Yc].as<double>(), c64[ci].as<long long>(), c32[ci].as<long long>(),
                    pl.offsets64.as<long long>(), pl.offsets32.as<long long>(), pl.kstart32.as<int>()};
    }
    KCHK(launch_quartet_schedule(qs, st));
    HF_CUDA(cudaMemcpyAsync(enn_dev, S->Ebuf.as<double>() + 300, sizeof(double), cudaMemcpyDeviceToDevice, st));
    HF_CUDA(cudaMemcpyAsync(enn_dev + 1, qbits_dev, sizeof(double), cudaMemcpyDeviceToDevice, st));
    unsigned char rbh[512];
    HF_CUDA(cudaMemcpyAsync(rbh, rb.p, 512, cudaMemcpyDeviceToHost, st));
    HF_CUDA(cudaStreamSynchronize(st));  // host sync: significant counts, quartet totals, E_nn
    const unsigned* nsig_h = (const unsigned*)rbh;
    const long long* totals_h = (const long long*)(rbh + 32);
    memcpy(&S->E_nn, rbh + 32 + 8 * 2 * kNumClasses, sizeof(double));
    memcpy(&S->Qmax, rbh + 32 + 8 * 2 * kNumClasses + 8, sizeof(double));
    for (int c = 0; c < kNumPairClasses; c++) S->class_count[c] = (int)nsig_h[c];
    for (int ci = 0; ci < kNumClasses; ci++) {
        S->plan[ci].n64 = totals_h[2 * ci];
        S->plan[ci].n32 = totals_h[2 * ci + 1];
    }
    // ket tables (field-major copies of each class's records in class-list order), headers in list order, and
    // bra lookup tables: one allocation, whose sizes follow from the counts just read
    Arena a4;
    const size_t rows = (size_t)X.maxpp;
    for (int c = 0; c < kNumPairClasses; c++) {
        const int n = S->class_count[c];
        if (n <= 0) continue;
        S->ket_stride[c] = ((long long)n + 31) / 32 * 32;
        a4.add(S->ket_tab[c], rows * S->ket_stride[c] * (9 * sizeof(double) + 9 * sizeof(float) + sizeof(float)));
        a4.add(S->class_hdr[c], sizeof(PairHdr) * (size_t)n);
    }
    for (auto& pl : S->plan) {
        if (pl.n64 > 0) a4.add(pl.chunk64, sizeof(int) * chunk_entries(pl.n64));
        if (pl.n32 > 0) a4.add(pl.chunk32, sizeof(int) * chunk_entries(pl.n32));
    }
    TRY(a4.commit(X.arena_tab));
    for (int c = 0; c < kNumPairClasses; c++) {
        const int n = S->class_count[c];
        if (n <= 0) continue;
        const long long stride = S->ket_stride[c];
        double* t64 = S->ket_tab[c].as<double>();
        float* t32 = (float*)(t64 + 9 * rows * stride);
        float* tB = t32 + 9 * rows * stride;
        KCHK(launch_ket_table(n, X.maxpp, stride, S->class_ids[c].as<int>(), S->pairs.as<PairHdr>(), S->prims64.p,
                              S->prims32.p, t64, t32, tB, st));
        KCHK(launch_gather_headers(n, S->class_ids[c].as<int>(), S->pairs.as<PairHdr>(), S->class_hdr[c].as<PairHdr>(),
                                   st));
    }
    ChunkTables ct{};
    for (int ci = 0; ci < kNumClasses; ci++) {
        auto& pl = S->plan[ci];
        const int nb = S->class_count[kEriClasses[ci].X];
        if (pl.n64 > 0) ct.t[ct.n++] = {nb, pl.offsets64.as<long long>(), pl.n64, chunk_entries(pl.n64), pl.chunk64.as<int>()};
        if (pl.n32 > 0) ct.t[ct.n++] = {nb, pl.offsets32.as<long long>(), pl.n32, chunk_entries(pl.n32), pl.chunk32.as<int>()};
    }
    KCHK(launch_chunk_bra(ct, st));
    HF_CUDA(cudaGetLastError());
    return HF_OK;
}

int hf::check_geometry_basis(const hf_geometry* g, const hf_basis* b, const hf_thresholds* th)
{
    if (!g || !b) return fail(HF_E_INVALID, "geometry or basis is NULL");
    if (g->n_atoms < 1 || !g->Z || !g->xyz) return fail(HF_E_INVALID, "geometry: empty or NULL arrays");
    if (b->n_shells < 1 || !b->atom || !b->l || !b->nprim || !b->exps || !b->coefs)
        return fail(HF_E_INVALID, "basis: empty or NULL arrays");
    for (int a = 0; a < g->n_atoms; a++) {
        if (g->Z[a] < 0) return fail(HF_E_INVALID, "geometry: negative nuclear charge");
        for (int x = 0; x < 3; x++)
            if (!isfinite(g->xyz[3 * a + x])) return fail(HF_E_INVALID, "geometry: non-finite coordinate");
    }
    long long np = 0;
    for (int s = 0; s < b->n_shells; s++) {
        if (b->atom[s] < 0 || b->atom[s] >= g->n_atoms) return fail(HF_E_INVALID, "basis: atom index out of range");
        if (b->l[s] == HF_SP_SHELL && !b->coefs_p)
            return fail(HF_E_INVALID, "basis: sp shell without p coefficients (coefs_p is NULL)");
        if (b->l[s] < 0 && b->l[s] != HF_SP_SHELL) return fail(HF_E_INVALID, "basis: negative angular momentum");
        if (b->l[s] > kMaxL) return fail(HF_E_UNSUPPORTED, "basis: l > 2 is not supported");
        if (b->nprim[s] < 1) return fail(HF_E_INVALID, "basis: shell without primitives");
        if (b->nprim[s] > kMaxPrim) return fail(HF_E_UNSUPPORTED, "basis: more than 8 primitives in a shell");
        np += b->nprim[s];
    }
    for (long long k = 0; k < np; k++) {
        if (!(b->exps[k] > 0.0) || !isfinite(b->exps[k])) return fail(HF_E_INVALID, "basis: exponent not positive");
        if (!isfinite(b->coefs[k])) return fail(HF_E_INVALID, "basis: non-finite coefficient");
    }
    if (b->coefs_p) {
        long long o = 0;
        for (int s = 0; s < b->n_shells; s++) {
            if (b->l[s] == HF_SP_SHELL)
                for (int k = 0; k < b->nprim[s]; k++)
                    if (!isfinite(b->coefs_p[o + k])) return fail(HF_E_INVALID, "basis: non-finite p coefficient");
            o += b->nprim[s];
        }
    }
    if (th) {
        if (!(th->schwarz_tau >= 0.0) || !(th->fp32_cutoff >= 0.0)) return fail(HF_E_INVALID, "thresholds: negative");
        if (!(th->prim_tau >= 0.0)) return fail(HF_E_INVALID, "thresholds: negative prim_tau");
    }
    return HF_OK;
}

// A basis with sp shells written as separate shells: each sp shell becomes an s shell (coefficients
// coefs) followed by a p shell (coefficients coefs_p) with the same exponents on the same atom, which
// keeps the basis-function order s, x, y, z of the sp shell.
struct ExpandedBasis {
    std::vector<int32_t> atom, l, nprim;
    std::vector<double> exps, coefs;
    hf_basis view{};
};

static const hf_basis* expand_sp_shells(const hf_basis* b, ExpandedBasis& e)
{
    bool any = false;
    for (int s = 0; s < b->n_shells; s++) any |= b->l[s] == HF_SP_SHELL;
    if (!any) return b;
    long long o = 0;
    for (int s = 0; s < b->n_shells; s++) {
        const int n = b->nprim[s];
        const int parts = b->l[s] == HF_SP_SHELL ? 2 : 1;
        for (int part = 0; part < parts; part++) {
            e.atom.push_back(b->atom[s]);
            e.l.push_back(b->l[s] == HF_SP_SHELL ? part : b->l[s]);
            e.nprim.push_back(n);
            const double* c = part == 1 ? b->coefs_p : b->coefs;
            for (int k = 0; k < n; k++) {
                e.exps.push_back(b->exps[o + k]);
                e.coefs.push_back(c[o + k]);
            }
        }
        o += n;
    }
    e.view.n_shells = (int32_t)e.l.size();
    e.view.atom = e.atom.data();
    e.view.l = e.l.data();
    e.view.nprim = e.nprim.data();
    e.view.exps = e.exps.data();
    e.view.coefs = e.coefs.data();
    e.view.coefs_p = nullptr;
    return &e.view;
}

int hf::create_system(hf_ctx* ctx, const hf_geometry* geom, const hf_basis* basis_in, const hf_thresholds* th,
                      std::shared_ptr<const ExponentTable> table, hf_system** out)
{
    TRY(check_geometry_basis(geom, basis_in, th));
    ExpandedBasis eb;
    const hf_basis* basis = expand_sp_shells(basis_in, eb);
    DeviceGuard g(ctx->device);
    hf_system* S = new hf_system();
    S->ctx = ctx;
    S->device = ctx->device;
    S->stream = ctx->stream;
    S->etab = std::move(table);
    if (th) S->th = *th;
    int rc = system_setup(S, geom, basis);
    if (rc != HF_OK) {
        cudaStreamSynchronize(ctx->stream);
        delete S;
        return rc;
    }
    ctx->n_systems++;
    *out = S;
    return HF_OK;
}

extern "C" {

int hf_system_create(hf_ctx* ctx, const hf_geometry* geom, const hf_basis* basis, const hf_thresholds* th,
                     hf_system** out)
{
    if (!ctx || !out) return fail(HF_E_INVALID, "hf_system_create: NULL ctx or output pointer");
    *out = nullptr;
    return create_system(ctx, geom, basis, th, nullptr, out);
}

void hf_system_destroy(hf_system* S)
{
    if (!S) return;
    hf_ctx* ctx = S->ctx;
    {
        DeviceGuard g(S->device);
        cudaStreamSynchronize(S->stream);
        delete S;
    }
    if (ctx && --ctx->n_systems == 0 && ctx->destroy_pending) ctx_release(ctx);
}

int hf_system_get_info(const hf_system* S, hf_system_info* info)
{
    if (!S || !info) return fail(HF_E_INVALID, "hf_system_get_info: NULL argument");
    memset(info, 0, sizeof(*info));
    info->n_atoms = S->n_atoms;
    info->n_shells = S->n_shells;
    info->n_bf = S->n_bf;
    info->n_electrons = S->n_electrons;
    info->n_pairs = S->n_pairs_all;
    for (int c = 0; c < kNumPairClasses; c++) info->n_significant_pairs += S->class_count[c];
    info->quartets_unscreened = S->quartets_total;
    for (int c = 0; c < kNumClasses; c++) {
        info->quartets_fp64 += S->plan[c].n64;
        info->quartets_fp32 += S->plan[c].n32;
    }
    info->E_nn = S->E_nn;
    info->Q_max = S->Qmax;
    long long bytes = 0;
    const DevBuf* bufs[] = {&S->sh_l, &S->sh_atom, &S->sh_bf0, &S->sh_nprim, &S->sh_prim0, &S->sh_exp, &S->sh_coef,
                            &S->atom_xyz, &S->atom_Z, &S->comp_norm, &S->pairs, &S->prims64, &S->prims32,
                            &S->pair_class, &S->S, &S->H, &S->P64, &S->P32, &S->Jt, &S->Kt, &S->F, &S->Ebuf,
                            &S->Qall, &S->staging_P, &S->staging_out, &S->hrec, &S->hB, &S->etab->tab};
    for (auto* b : bufs) bytes += b->bytes;
    for (int c = 0; c < kNumPairClasses; c++)
        bytes += S->class_ids[c].bytes + S->class_q[c].bytes + S->ket_tab[c].bytes + S->class_hdr[c].bytes;
    for (int c = 0; c < kNumClasses; c++)
        bytes += S->plan[c].offsets64.bytes + S->plan[c].offsets32.bytes + S->plan[c].kstart32.bytes +
                 S->plan[c].chunk64.bytes + S->plan[c].chunk32.bytes;
    info->device_bytes = bytes;
    return HF_OK;
}

int hf_one_electron(hf_system* S, double* Sout, double* Hout, int flags)
{
    if (!S) return fail(HF_E_INVALID, "hf_one_electron: NULL system");
    DeviceGuard g(S->ctx->device);
    const size_t bytes = (size_t)S->n_bf * S->n_bf * sizeof(double);
    const cudaMemcpyKind kind = (flags & HF_PTR_DEVICE) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    cudaStream_t st = S->ctx->stream;
    if (Sout) HF_CUDA(cudaMemcpyAsync(Sout, S->S.p, bytes, kind, st));
    if (Hout) HF_CUDA(cudaMemcpyAsync(Hout, S->H.p, bytes, kind, st));
    HF_CUDA(cudaStreamSynchronize(st));
    return HF_OK;
}

// Accumulators of one build: the system's Jt / Kt (one copy shared by every block, updated with FP64
// atomics), or fock_copies zeroed copies of each, block b writing copy b % fock_copies, summed into
// Jt / Kt after the ERI launches (the GPU analogue of the paper's private Fock matrices).
static int begin_accumulate(hf_system& X, EriArgs& a, cudaStream_t st)
{
    const size_t NN = (size_t)X.n_bf * X.n_bf;
    if (X.fock_copies > 1) {
        HF_CUDA(cudaMemsetAsync(X.copies.p, 0, 2 * (size_t)X.fock_copies * NN * sizeof(double), st));
        a.Jt = X.copies.as<double>();
        a.Kt = a.Jt + (size_t)X.fock_copies * NN;
        a.n_copies = X.fock_copies;
        a.copy_stride = (long long)NN;
    } else {
        HF_CUDA(cudaMemsetAsync(X.Jt.p, 0, NN * sizeof(double), st));
        HF_CUDA(cudaMemsetAsync(X.Kt.p, 0, NN * sizeof(double), st));
        a.Jt = X.Jt.as<double>();
        a.Kt = X.Kt.as<double>();
        a.n_copies = 1;
        a.copy_stride = 0;
    }
    return HF_OK;
}

static int end_accumulate(hf_system& X, cudaStream_t st)
{
    if (X.fock_copies <= 1) return HF_OK;
    const long long NN = (long long)X.n_bf * X.n_bf;
    const double* c = X.copies.as<double>();
    KCHK(launch_sum_copies(X.fock_copies, NN, c, X.Jt.as<double>(), X.ctx->num_sms, st));
    KCHK(launch_sum_copies(X.fock_copies, NN, c + (size_t)X.fock_copies * NN, X.Kt.as<double>(), X.ctx->num_sms, st));
    return HF_OK;
}

int hf_system_set_fock_copies(hf_system* S, int32_t copies)
{
    if (!S) return fail(HF_E_INVALID, "hf_system_set_fock_copies: NULL system");
    if (copies < 1 || copies > 4096) return fail(HF_E_INVALID, "hf_system_set_fock_copies: copies must be 1..4096");
    DeviceGuard g(S->ctx->device);
    HF_CUDA(cudaStreamSynchronize(S->ctx->stream));
    if (copies == 1) {
        S->copies.release();
        S->fock_copies = 1;
        return HF_OK;
    }
    const size_t NN = (size_t)S->n_bf * S->n_bf;
    S->copies.release();
    S->fock_copies = 1;
    if (S->copies.alloc(2 * (size_t)copies * NN * sizeof(double)) != HF_OK) {
        cudaGetLastError();
        return fail(HF_E_NOMEM, "hf_system_set_fock_copies: cannot allocate the accumulator copies");
    }
    S->fock_copies = copies;
    return HF_OK;
}

}  // extern "C"

constexpr int kBeside32 = 2;  // blocks per SM of an FP32 launch beside FP64 ones

// One class launch of a build.
struct ClassLaunch {
    int ci, prec, use_f32;
    Fp64Method method;
    bool warp;   // Hermite warp kernel
    int lanes;   // lanes per quartet (thread kernels), parts per quartet (warp kernel)
    int rounds;  // Hermite thread kernel: rounds per sorted window; warp kernel: > 1 for groups of quartets
    int grid;
    double est;  // estimated device time, in operations of the whole GPU
};

// The per-class ERI launches shared by hf_fock_build, hf_fock_build_partial and hf_fock_build_noalloc.
//
// Small systems: a class with a few hundred quartets lasts as long as its slowest quartet whatever the GPU
// could do beside it, and the classes' launches, one after another, add those latencies up (one water: 21
// launches of 0.1 to 5.8 ms each for 0.05 ms of arithmetic).  The launches are independent (they only add
// into J and K), so they are spread over the side streams, the longest first (by the larger of the class's
// share of the GPU's rate and the latency of one quartet), each to the stream with the least work so far.
// Large systems gain the same way at each class's tail.
int hf::launch_eri_classes(hf_system* S, EriArgs a, int shard, int n_shards, int flags, cudaEvent_t* ev,
                           unsigned long long* prim_count)
{
    hf_ctx* ctx = S->ctx;
    hf_system& X = *S;
    a.pairs = S->pairs.as<PairHdr>();
    a.prims64 = S->prims64.p;
    a.prims32 = S->prims32.p;
    a.N = S->n_bf;
    a.boys64 = ctx->boys64.as<double>();
    a.boys32 = ctx->boys32.as<float>();
    a.prim_tau = S->th.prim_tau;
    a.herm = S->herm;
    ClassLaunch todo[2 * kNumClasses];
    int n_todo = 0;
    // primitive quartets of a quartet (about 0.4 of them survive the primitive threshold) and the time of the whole
    // build at 1.1 TFLOP/s
    const double prims = (S->th.prim_tau > 0.0 ? 0.4 : 1.0) * X.maxpp * X.maxpp;
    double t_all = 0.0, t_all32 = 0.0;
    for (int ci = 0; ci < kNumClasses; ci++) {
        const double n = (double)S->plan[ci].n64 + ((flags & HF_FP64_ONLY) ? (double)S->plan[ci].n32 : 0.0);
        t_all += n / n_shards * (kEriClasses[ci].prim_flops_h * prims + kEriClasses[ci].cont_flops_h) / 1.1e12;
        if (!(flags & HF_FP64_ONLY))
            t_all32 += (double)S->plan[ci].n32 / n_shards * (kEriClasses[ci].prim_flops * prims + kEriClasses[ci].cont_flops) / 1.0e13;
    }
    for (int ci = 0; ci < kNumClasses; ci++)
        for (int prec = 0; prec < 2; prec++) {
            const long long n = prec ? S->plan[ci].n32 : S->plan[ci].n64;
            const long long nq = n * (shard + 1) / n_shards - n * shard / n_shards;
            const EriClassEntry& cl = kEriClasses[ci];
            ClassLaunch c{ci, prec, prec && !(flags & HF_FP64_ONLY), fp64_method(ci, flags), false, 1, 1, 0, 0.0};
            // a class too small to fill the GPU with one thread per quartet
            const bool small = !c.use_f32 && nq < (long long)ctx->num_sms * 256;
            const long long windows_min = (long long)ctx->num_sms * 4;
            double ops = (double)cl.prim_flops * prims + cl.cont_flops;
            if (!c.use_f32 && c.method == Fp64Method::kHerm) {
                ops = (double)cl.prim_flops_h * prims + cl.cont_flops_h;
                // One thread per quartet wastes the least, but lasts as long as one lane needs for a quartet
                // (about 0.65 FP64 instructions an operation, 64 clocks each, three warps sharing a scheduler): fine
                // while that is half of the whole build, which the other classes fill.  Otherwise a small launch
                // shares each quartet among a lane group or a warp.  Against "small" alone: split-valence 10 waters
                // 7.0 -> 5.1 ms, 4 waters unscreened 10.9 -> 10.3 ms (a quarter or twice of the half: within 1%).
                const double lat = ops * 0.65 * 64.0 * 3.0 / 2.0e9;
                const bool fits = cl.launch_herm && lat <= 0.5 * t_all;
                c.warp = !cl.launch_herm || (small && !fits && cl.launch_hermw);
                if (c.warp) {
                    // parts: quartets fewer than four warps per SM take one warp per batch of 32 primitive quartets
                    const long long batches = ((long long)X.maxpp * X.maxpp + 31) / 32;
                    c.lanes = (int)std::max<long long>(1, std::min(batches, (long long)ctx->num_sms * 4 / std::max<long long>(nq, 1)));
                    // groups of quartets per warp once there are eight warps per SM without them
                    if (nq >= (long long)ctx->num_sms * 64) c.rounds = 2;
                } else {
                    if (small && !fits) c.lanes = cl.herm_lanes;
                    // sorted windows: as many rounds as keep four windows per SM and the same latency bound (without
                    // the sort 32 waters 812 -> 831 ms and split-valence 10 waters 5.35 -> 5.96; one window per SM
                    // 13 waters 70 -> 75)
                    while (c.lanes == 1 && c.rounds < kSortRounds && nq >= windows_min * 64 * c.rounds &&
                           2 * c.rounds * lat <= 0.5 * t_all)
                        c.rounds *= 2;
                    const long long per_block = (long long)(kEriThreads / c.lanes) * c.rounds;
                    c.grid = (int)std::min<long long>((nq + per_block - 1) / per_block, 1 << 20);
                }
            } else {
                // shares each quartet's primitive work among a lane group (shorter latency, same result)
                if (small) c.lanes = cl.lanes;
                c.grid = (int)std::min<long long>((nq * c.lanes + kEriThreads - 1) / kEriThreads, (long long)ctx->num_sms * 16);
            }
            // one quartet's operations run in one lane (warp), 1 / (64 lanes SMs) of the GPU at a time
            c.est = std::max((double)nq, 64.0 * ctx->num_sms / (c.warp ? 32 * c.lanes : c.lanes)) * ops / (c.use_f32 ? 32.0 : 1.0);
            if (nq > 0 || ev) todo[n_todo++] = c;
        }
    const bool forked = !ev && n_todo > 1;
    double load[kSideStreams] = {};
    SideStreams side(ctx);
    if (forked) {
        std::sort(todo, todo + n_todo, [](const ClassLaunch& x, const ClassLaunch& y) { return x.est > y.est; });
        TRY(side.fork());
    }
    // The FP64 kernels keep the FP64 pipe busy and leave nine of ten issue slots free; the FP32 kernels of a mixed
    // build need those slots and next to no FP64.  On one SM at the same time the shorter part costs little, but
    // blocks of equal priority run one kernel after the other.  So the FP32 launches go to the stream of higher
    // priority, with few enough persistent blocks that FP64 blocks fit beside them: kBeside32 per SM while the FP32
    // part is the shorter one, all the SM holds otherwise.  (The quartets above an FP32 cutoff keep about twice the
    // primitive quartets that t_all assumes, and those below it fewer: 64 waters, FP64 955 ms, FP32 300 ms alone,
    // estimated 370 and 410.)  Measured: mixed 64 waters 1,245 -> 1,150 ms, a 24-water difference build 103 -> 94 ms;
    // 2 to 8 blocks per SM within 1%.
    const bool beside = forked && t_all32 > 0.0 && t_all32 < 2.0 * t_all;
    cudaError_t err = cudaSuccess;
    for (int t = 0; t < n_todo && err == cudaSuccess; t++) {
        const ClassLaunch& c = todo[t];
        const auto& pl = S->plan[c.ci];
        const int Xc = kEriClasses[c.ci].X, Yc = kEriClasses[c.ci].Y;
        cudaStream_t st = ctx->stream;
        int grid = c.grid;
        if (beside && c.use_f32) {
            st = ctx->fast;
            grid = std::min(grid, ctx->num_sms * kBeside32);
        } else if (forked) {
            const int i = (int)(std::min_element(load, load + kSideStreams) - load);
            load[i] += c.est;
            st = ctx->side[i];
        }
        a.bra = S->class_ids[Xc].as<int>();
        a.ket = S->class_ids[Yc].as<int>();
        a.bhdr = S->class_hdr[Xc].as<PairHdr>();
        a.khdr = S->class_hdr[Yc].as<PairHdr>();
        a.n_bra = S->class_count[Xc];
        a.same = Xc == Yc;
        const long long n = c.prec ? pl.n32 : pl.n64;
        a.q_begin = n * shard / n_shards;
        a.n_quartets = n * (shard + 1) / n_shards;
        if (ev) err = cudaEventRecord(ev[4 * c.ci + 2 * c.prec], st);
        a.prim_count = prim_count ? prim_count + 2 * c.ci + c.prec : nullptr;
        if (a.n_quartets > a.q_begin && err == cudaSuccess) {
            a.offsets = c.prec ? pl.offsets32.as<long long>() : pl.offsets64.as<long long>();
            a.kstart = c.prec ? pl.kstart32.as<int>() : nullptr;
            a.chunk = c.prec ? pl.chunk32.as<int>() : pl.chunk64.as<int>();
            a.kt = nullptr;
            a.ktB = nullptr;
            a.kstride = 0;
            if (X.ket_tab[Yc].p) {
                const long long st_ = X.ket_stride[Yc];
                const double* t64 = X.ket_tab[Yc].as<double>();
                const float* t32 = (const float*)(t64 + 9 * (size_t)X.maxpp * st_);
                a.kt = c.use_f32 ? (const void*)t32 : (const void*)t64;
                a.ktB = t32 + 9 * (size_t)X.maxpp * st_;
                a.kstride = st_;
            }
            // FP64 launches run each warp's window of quartets sorted by staircase length (64 waters:
            // 2% faster); the FP32 kernels, bound by latency rather than a pipe, ran 10% slower with it
            // and are compiled without it
            a.sort_work = c.use_f32 ? 0 : 1;
            a.rounds = c.rounds;
            const EriClassEntry& cl = kEriClasses[c.ci];
            if (c.use_f32 || c.method == Fp64Method::kObaraSaika)
                cl.launch(a, c.use_f32, grid, kEriThreads, st, c.lanes);
            else if (c.method == Fp64Method::kRys)
                cl.launch_rys(a, 0, c.grid, kEriThreads, st, c.lanes);
            else if (c.warp)
                cl.launch_hermw(a, st, c.rounds > 1, c.lanes);
            else
                cl.launch_herm(a, c.grid, st, c.lanes);
            err = cudaGetLastError();
        }
        if (ev && err == cudaSuccess) err = cudaEventRecord(ev[4 * c.ci + 2 * c.prec + 1], st);
    }
    const int rc = side.join();
    if (err == cudaSuccess && rc != HF_OK) return rc;
    return err == cudaSuccess ? HF_OK : cuda_status(err, "ERI class launch");
}

extern "C" {

int hf_fock_build(hf_system* S, const double* P, double* F, double* J, double* K, double* E_elec, hf_stats* stats,
                  int flags)
{
    if (!S || !P) return fail(HF_E_INVALID, "hf_fock_build: NULL system or density");
    DeviceGuard g(S->ctx->device);
    hf_ctx* ctx = S->ctx;
    hf_system& X = *S;
    cudaStream_t st = ctx->stream;
    const int N = S->n_bf;
    const size_t NN = (size_t)N * N;
    const bool dev = (flags & HF_PTR_DEVICE) != 0;
    const bool timing = (flags & HF_TIMING) != 0 && stats;
    // 1. density in, check, raw-normalised copies.  The check's flag stays on the device: the ERI,
    // assembly and energy kernels do nothing when it is set, and the host reads it once, at the end.
    const double* dP = P;
    if (!dev) {
        HF_CUDA(cudaMemcpyAsync(X.staging_P.p, P, NN * sizeof(double), cudaMemcpyHostToDevice, st));
        dP = X.staging_P.as<double>();
    }
    if (timing) HF_CUDA(cudaEventRecord(ctx->ev[4 * kNumClasses], st));
    HF_CUDA(cudaMemsetAsync(X.bad.p, 0, sizeof(int), st));
    KCHK(launch_scale_density(N, dP, S->comp_norm.as<double>(), S->P64.as<double>(),
                              S->P32.p ? S->P32.as<float>() : nullptr, X.bad.as<int>(), st));
    // 2. ERI + digestion, one launch per class and precision
    EriArgs a;
    memset(&a, 0, sizeof(a));
    TRY(begin_accumulate(X, a, st));
    if (timing) HF_CUDA(cudaEventRecord(ctx->ev[4 * kNumClasses + 1], st));
    a.P64 = S->P64.as<double>();
    a.P32 = S->P32.p ? S->P32.as<float>() : nullptr;
    a.bad = X.bad.as<int>();
    if (stats) HF_CUDA(cudaMemsetAsync(X.prim_count.p, 0, sizeof(unsigned long long) * 2 * kNumClasses, st));
    TRY(launch_eri_classes(S, a, 0, 1, flags, timing ? ctx->ev : nullptr,
                           stats ? X.prim_count.as<unsigned long long>() : nullptr));
    TRY(end_accumulate(X, st));
    if (timing) HF_CUDA(cudaEventRecord(ctx->ev[4 * kNumClasses + 2], st));
    // 3. symmetrise and assemble (skipped on the device when the density was rejected)
    double* dF = dev && F ? F : S->F.as<double>();
    double* dJ = dev ? J : (J ? X.staging_out.as<double>() : nullptr);
    double* dK = dev ? K : (K ? X.staging_out.as<double>() + NN : nullptr);
    KCHK(launch_assemble(N, S->Jt.as<double>(), S->Kt.as<double>(), S->comp_norm.as<double>(), S->H.as<double>(), dJ,
                         dK, dF, X.bad.as<int>(), st));
    if (E_elec) KCHK(launch_energy(N, dP, S->H.as<double>(), dF, S->Ebuf.as<double>(), S->Ebuf.as<double>() + 256, st));
    if (timing) HF_CUDA(cudaEventRecord(ctx->ev[4 * kNumClasses + 3], st));
    int bad = 0;
    double e_host = 0.0;
    HF_CUDA(cudaMemcpyAsync(&bad, X.bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    if (E_elec) HF_CUDA(cudaMemcpyAsync(&e_host, S->Ebuf.as<double>() + 256, sizeof(double), cudaMemcpyDeviceToHost, st));
    HF_CUDA(cudaStreamSynchronize(st));
    HF_CUDA(cudaGetLastError());
    if (bad) return fail(HF_E_INVALID, "hf_fock_build: density is not finite or not symmetric");
    if (!dev) {  // host outputs are written only once the density is known to be valid
        if (F) HF_CUDA(cudaMemcpyAsync(F, dF, NN * sizeof(double), cudaMemcpyDeviceToHost, st));
        if (J) HF_CUDA(cudaMemcpyAsync(J, dJ, NN * sizeof(double), cudaMemcpyDeviceToHost, st));
        if (K) HF_CUDA(cudaMemcpyAsync(K, dK, NN * sizeof(double), cudaMemcpyDeviceToHost, st));
        HF_CUDA(cudaStreamSynchronize(st));
    }
    if (E_elec) *E_elec = e_host;
    if (stats) {
        unsigned long long pc[2 * kNumClasses];
        HF_CUDA(cudaMemcpy(pc, X.prim_count.p, sizeof(pc), cudaMemcpyDeviceToHost));
        memset(stats, 0, sizeof(*stats));
        stats->quartets_unscreened = S->quartets_total;
        for (int ci = 0; ci < kNumClasses; ci++) {
            const auto& pl = S->plan[ci];
            stats->class_quartets_fp64[ci] = pl.n64;
            stats->class_quartets_fp32[ci] = pl.n32;
            stats->quartets_fp64 += pl.n64;
            stats->quartets_fp32 += pl.n32;
            stats->prim_quartets_fp64 += (int64_t)pc[2 * ci];
            stats->prim_quartets_fp32 += (int64_t)pc[2 * ci + 1];
            const EriClassEntry& cl = kEriClasses[ci];
            const Fp64Method m = fp64_method(ci, flags);
            const bool herm = m == Fp64Method::kHerm;
            const double pf64 = herm ? cl.prim_flops_h : m == Fp64Method::kRys ? cl.prim_flops_rys : cl.prim_flops;
            const double cf64 = herm ? cl.cont_flops_h : cl.cont_flops;
            const bool f64 = (flags & HF_FP64_ONLY) != 0;  // else FP32 launches, which are Obara-Saika
            stats->class_flops_fp64[ci] = pf64 * (double)pc[2 * ci] + cf64 * (double)pl.n64;
            stats->class_flops_fp32[ci] = (f64 ? pf64 : cl.prim_flops) * (double)pc[2 * ci + 1] +
                                          (f64 ? cf64 : cl.cont_flops) * (double)pl.n32;
            stats->flops_fp64 += stats->class_flops_fp64[ci];
            stats->flops_fp32 += stats->class_flops_fp32[ci];
            stats->kernels_launched += (pl.n64 > 0) + (pl.n32 > 0);
            if (timing) {
                cudaEventElapsedTime(&stats->ms_class_fp64[ci], ctx->ev[4 * ci], ctx->ev[4 * ci + 1]);
                cudaEventElapsedTime(&stats->ms_class_fp32[ci], ctx->ev[4 * ci + 2], ctx->ev[4 * ci + 3]);
            }
        }
        stats->kernels_launched += 2 + (E_elec ? 2 : 0) + (X.fock_copies > 1 ? 2 : 0);  // density scaling,
                                                                                    // assembly, energy, copy sums
        if (timing) {
            cudaEventElapsedTime(&stats->ms_eri, ctx->ev[4 * kNumClasses + 1], ctx->ev[4 * kNumClasses + 2]);
            cudaEventElapsedTime(&stats->ms_total, ctx->ev[4 * kNumClasses], ctx->ev[4 * kNumClasses + 3]);
        }
    }
    return HF_OK;
}


// One shard of the Fock build: the quartets [n s / S, n (s+1) / S) of every class launch.
int hf_fock_build_partial(hf_system* S, const double* P, int shard, int n_shards, double* J, double* K, int flags)
{
    if (!S || !P || !J || !K) return fail(HF_E_INVALID, "hf_fock_build_partial: NULL argument");
    if (n_shards < 1 || shard < 0 || shard >= n_shards) return fail(HF_E_INVALID, "hf_fock_build_partial: bad shard");
    DeviceGuard g(S->ctx->device);
    hf_ctx* ctx = S->ctx;
    hf_system& X = *S;
    cudaStream_t st = ctx->stream;
    const int N = S->n_bf;
    const size_t NN = (size_t)N * N;
    const bool dev = (flags & HF_PTR_DEVICE) != 0;
    const double* dP = P;
    if (!dev) {
        HF_CUDA(cudaMemcpyAsync(X.staging_P.p, P, NN * sizeof(double), cudaMemcpyHostToDevice, st));
        dP = X.staging_P.as<double>();
    }
    HF_CUDA(cudaMemsetAsync(X.bad.p, 0, sizeof(int), st));
    KCHK(launch_scale_density(N, dP, S->comp_norm.as<double>(), S->P64.as<double>(),
                              S->P32.p ? S->P32.as<float>() : nullptr, X.bad.as<int>(), st));
    EriArgs a;
    memset(&a, 0, sizeof(a));
    TRY(begin_accumulate(X, a, st));
    a.P64 = S->P64.as<double>();
    a.P32 = S->P32.p ? S->P32.as<float>() : nullptr;
    a.bad = X.bad.as<int>();
    if ((flags & HF_DENSITY_SCREEN) && S->th.schwarz_tau > 0.0) {
        if (!X.dsh.p) TRY(X.dsh.alloc(sizeof(float) * (size_t)S->n_shells * S->n_shells));
        KCHK(launch_shell_block_max(S->n_shells, N, S->sh_l.as<int>(), S->sh_bf0.as<int>(), dP, X.dsh.as<float>(),
                                    st));
        a.dsh = X.dsh.as<float>();
        a.n_sh = S->n_shells;
        a.dtau = (float)S->th.schwarz_tau;
    }
    TRY(launch_eri_classes(S, a, shard, n_shards, flags, nullptr, nullptr));
    TRY(end_accumulate(X, st));
    // J and K of this shard (no H): the assembly kernel's F output is only scratch here
    double* dJ = dev ? J : X.staging_out.as<double>();
    double* dK = dev ? K : X.staging_out.as<double>() + NN;
    KCHK(launch_assemble(N, S->Jt.as<double>(), S->Kt.as<double>(), S->comp_norm.as<double>(), S->H.as<double>(), dJ,
                         dK, S->F.as<double>(), X.bad.as<int>(), st));
    int bad = 0;
    HF_CUDA(cudaMemcpyAsync(&bad, X.bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    HF_CUDA(cudaStreamSynchronize(st));
    if (bad) return fail(HF_E_INVALID, "hf_fock_build_partial: density is not finite or not symmetric");
    if (!dev) {
        HF_CUDA(cudaMemcpyAsync(J, dJ, NN * sizeof(double), cudaMemcpyDeviceToHost, st));
        HF_CUDA(cudaMemcpyAsync(K, dK, NN * sizeof(double), cudaMemcpyDeviceToHost, st));
        HF_CUDA(cudaStreamSynchronize(st));
    }
    return HF_OK;
}

// F = H + J - K/2 (and E_elec) from J and K summed over the shards of a sharded build.
int hf_fock_assemble(hf_system* S, const double* P, const double* J, const double* K, double* F, double* E_elec,
                     int flags)
{
    if (!S || !J || !K || !F) return fail(HF_E_INVALID, "hf_fock_assemble: NULL system, J, K or F");
    if (E_elec && !P) return fail(HF_E_INVALID, "hf_fock_assemble: the energy needs the density P");
    DeviceGuard g(S->ctx->device);
    hf_system& X = *S;
    cudaStream_t st = S->ctx->stream;
    const int N = S->n_bf;
    const size_t NN = (size_t)N * N;
    const bool dev = (flags & HF_PTR_DEVICE) != 0;
    const double *dJ = J, *dK = K, *dP = P;
    double* dF = dev ? F : S->F.as<double>();
    if (!dev) {  // staging: J and K in staging_out, P in staging_P
        HF_CUDA(cudaMemcpyAsync(X.staging_out.p, J, NN * sizeof(double), cudaMemcpyHostToDevice, st));
        HF_CUDA(cudaMemcpyAsync(X.staging_out.as<double>() + NN, K, NN * sizeof(double), cudaMemcpyHostToDevice, st));
        dJ = X.staging_out.as<double>();
        dK = dJ + NN;
        if (P) {
            HF_CUDA(cudaMemcpyAsync(X.staging_P.p, P, NN * sizeof(double), cudaMemcpyHostToDevice, st));
            dP = X.staging_P.as<double>();
        }
    }
    HF_CUDA(cudaMemsetAsync(X.bad.p, 0, sizeof(int), st));
    KCHK(launch_fock_from_jk((long long)NN, S->H.as<double>(), dJ, dK, dF, X.bad.as<int>(), st));
    if (E_elec) KCHK(launch_energy(N, dP, S->H.as<double>(), dF, S->Ebuf.as<double>(), S->Ebuf.as<double>() + 256, st));
    int bad = 0;
    double e_host = 0.0;
    HF_CUDA(cudaMemcpyAsync(&bad, X.bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    if (E_elec) HF_CUDA(cudaMemcpyAsync(&e_host, S->Ebuf.as<double>() + 256, sizeof(double), cudaMemcpyDeviceToHost, st));
    HF_CUDA(cudaStreamSynchronize(st));
    if (bad) return fail(HF_E_INVALID, "hf_fock_assemble: J or K is not finite");
    if (!dev) {
        HF_CUDA(cudaMemcpyAsync(F, dF, NN * sizeof(double), cudaMemcpyDeviceToHost, st));
        HF_CUDA(cudaStreamSynchronize(st));
    }
    if (E_elec) *E_elec = e_host;
    return HF_OK;
}
}  // extern "C"
