// Internal declarations of the GB300 direct-SCF Fock-build library.
// Not part of the C-ABI (that is include/hf.h).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/hf.h"

namespace hf {

constexpr int kMaxL = 2;
constexpr int kNumPairClasses = 6;  // ss ps pp ds dp dd
constexpr int kNumClasses = 21;     // (X|Y), X >= Y
constexpr int kChunkShift = 10;      // quartets per entry of the bra lookup tables: 1024
constexpr int kMaxPrim = 8;         // primitives per shell accepted by the library
constexpr int kSideStreams = 8;     // streams the class launches of one build are spread over

// One significant shell pair, oriented so that l_A >= l_B.
struct PairHdr {
    int A, B;          // shell ids
    int bfA, bfB;      // first basis function of shells A and B
    int prim0, nprim;  // primitive-pair records [prim0, prim0 + nprim)
    double ABx, ABy, ABz;
    double Q;          // Cauchy-Schwarz bound sqrt(max |(mu nu|mu nu)|)
    float ABfx, ABfy, ABfz;  // A - B in FP32 (the FP32 kernels' horizontal step uses no FP64 instruction)
};

// Primitive-pair record of the Hermite-accumulator kernels: P, K (2p)^-W with the prefactor K of PrimPair,
// p = a + b and W = l_A + l_B, u = 2b, v = 2p, and the type of p in the exponent table.  Four 16-byte loads.
struct alignas(16) HermPair {
    double Px, Py, Pz;
    double K;
    double u, v;
    int type, pad[3];
};

// What the Hermite-accumulator kernels read of a system: records (HermPair of pair t at t maxpp, sorted by
// bound), their bounds in an array of their own (the screening loops read nothing else), and the exponent table
// (nullptr: evaluate directly).
struct HermView {
    const HermPair* rec;
    const float* B;
    const double2* etab;
    int ntype;
};
constexpr double kPairPrefactor = 5.914967172795613;  // sqrt(2) pi^(5/4): two pairs' product is 2 pi^(5/2)
constexpr double kNuclearPrefactor = 1.0622519320271968;  // 2 pi / kPairPrefactor (as rounded)
constexpr int kHermMaxTypes = 1448;  // 32 MB of exponent table

struct EriArgs {
    const PairHdr* pairs;
    const void* prims64;  // PrimPair<double>[]
    const void* prims32;  // PrimPair<float>[]
    const int* bra;       // bra pair ids (one class, sorted by Q descending)
    const int* ket;       // ket pair ids
    const long long* offsets;  // [n_bra + 1] exclusive prefix of quartets per bra
    const int* kstart;         // [n_bra] first ket of each bra (nullptr: 0)
    int n_bra;
    int same;                  // bra and ket lists are the same list
    long long n_quartets;
    int N;
    const double* P64;  // density in the library's raw component normalisation
    const float* P32;
    double* Jt;
    double* Kt;
    const double* boys64;
    const float* boys32;
    double prim_tau;                  // skip primitive quartets with B_ab * B_cd < prim_tau
    unsigned long long* prim_count;   // evaluated primitive quartets (nullptr: not counted)
    long long q_begin;                // first quartet of this launch (quartets [q_begin, n_quartets))
    const float* dsh;                 // [n_sh x n_sh] max |P| per shell block (nullptr: no density screening)
    int n_sh;
    float dtau;                       // density-weighted screening threshold
    const int* chunk;                 // [c] bra of quartet min(c << kChunkShift, n_quartets_all - 1)
                                      // (nullptr: each quartet's bra by binary search over all bras)
    int n_copies;                     // > 1: block b accumulates into copy b % n_copies of Jt / Kt
    long long copy_stride;            // doubles between copies
    const int* bad;                   // density-check flag: the kernel does nothing when *bad != 0
    const void* kt;                   // ket table of the launch's ket class and precision (field-major records
                                      // in class-list order, see KetSoa): read by the FP32 and Rys kernels; the
                                      // FP64 Obara-Saika kernels read each pair's own records
    const float* ktB;                 // primitive-pair bounds of the ket table
    long long kstride;                // kets per field row of the ket table
    const PairHdr* bhdr;              // headers of the bra list in list order (bhdr[b] = pairs[bra[b]])
    const PairHdr* khdr;              // headers of the ket list in list order (khdr[k] = pairs[ket[k]])
    HermView herm;
    int rounds;                       // Hermite thread kernels: rounds per sorted window (1: launch order)
    int sort_work;                    // Obara-Saika kernels, 1: each warp runs its window of quartets sorted by staircase length
};

struct SchwarzArgs {
    const PairHdr* pairs;
    HermView herm;
    const int* ids;       // pair ids of one diagonal class
    int n;
    double* Q;            // [pair id] output bound
    const double* boys64;
    double* Bprim;        // [primitive pair] output bound of each primitive pair
    int items;            // threads per pair: 1 + the largest primitive-pair count
};

// One-electron matrices of one pair class (onee_herm.cuh).
struct OneEArgs {
    const PairHdr* pairs;
    const int* ids;  // pair ids of the class
    int n, n_atoms, N;
    const int* nprim;
    const int* prim0;
    const double* exps;
    const double* cn;
    const double* xyz;
    const double* Z;
    const double* comp_norm;
    const double* boys64;
    HermView herm;
    double* S;
    double* H;
};

int launch_one_electron_class(int X, const OneEArgs& a, cudaStream_t s);

// One molecule's view of one class in a batched build.
struct MolClass {
    const PairHdr* bhdr;  // headers of the bra and ket lists in list order
    const PairHdr* khdr;
    HermView herm;
    const long long* offsets;  // [n_bra + 1]
    int n_bra;
    int same;
    int N;
    int pad;
    const double* P64;
    double* Jt;
    double* Kt;
};

struct BatchArgs {
    const MolClass* mols;        // [n_mol]
    const long long* mol_off;    // [n_mol + 1] exclusive prefix of this class's quartets per molecule
    int n_mol;
    int chunk;                   // quartets per work-queue grab (per warp)
    long long n_total;
    unsigned long long* counter; // work-queue head, zero at launch
    double prim_tau;
    const double* boys64;
};

struct EriClassEntry {
    int X, Y, L;
    // Hermite-accumulator kernels (the FP64 default): the thread kernel (nullptr: the class has none), the warp
    // kernel (nullptr: none; group 1: several quartets per warp), operations per primitive and per contracted quartet
    int prim_flops_h, cont_flops_h;
    void (*launch_herm)(const EriArgs&, int grid, cudaStream_t, int lanes);
    int herm_lanes;  // lanes per quartet of the thread kernel in small launches
    void (*launch_hermw)(const EriArgs&, cudaStream_t, int group, int nparts);
    int (*prepare)();             // sets the kernels' shared-memory limits once per device
    size_t (*local_bytes_h)();
    int batch_warp;               // 1: the batched kernel is one warp per block
    // Obara-Saika kernels: FP32, and FP64 with HF_OBARA_SAIKA
    int prim_flops;  // per primitive quartet (setup + Boys + VRR + accumulation)
    int cont_flops;  // per contracted quartet (HRR + digestion)
    void (*launch)(const EriArgs&, int use_f32, int grid, int block, cudaStream_t, int lanes);
    void (*launch_schwarz)(const SchwarzArgs&, int block, cudaStream_t);
    const char* name;
    void (*launch_batch)(const BatchArgs&, int grid, int block, cudaStream_t);
    size_t (*local_bytes)();  // largest per-thread local memory of the class's kernels
    int lanes;                // lanes that share one shell quartet in the ERI kernels
    // Rys-quadrature variant (classes with L >= 6; nullptr otherwise): FP64 launches with ket tables
    void (*launch_rys)(const EriArgs&, int use_f32, int grid, int block, cudaStream_t, int lanes);
    int prim_flops_rys;       // per primitive quartet (setup + roots + 2D recurrences + accumulation)
    size_t (*local_bytes_rys)();
};
extern const EriClassEntry kEriClasses[kNumClasses];

// Method of the FP64 launches of class ci under these build flags: Obara-Saika with HF_OBARA_SAIKA, Rys
// quadrature with HF_RYS for the classes that have it, else Hermite accumulators.
enum class Fp64Method { kHerm, kObaraSaika, kRys };
inline Fp64Method fp64_method(int ci, int flags)
{
    if (flags & HF_OBARA_SAIKA) return Fp64Method::kObaraSaika;
    return (flags & HF_RYS) && kEriClasses[ci].launch_rys ? Fp64Method::kRys : Fp64Method::kHerm;
}

// Launches the ERI class kernels of one build: for every class and precision, the quartets
// [n shard / n_shards, n (shard + 1) / n_shards) of its n screened quartets (shard 0 of 1 is the
// whole build).  `a` carries the fields common to every launch (density, accumulators, tables,
// screening and flag pointers); the per-class fields are filled here.  flags: HF_FP64_ONLY.
// The launches run concurrently on the context's side streams, between an event recorded on the context's
// stream and one it waits for; with ev they run one after another on the context's stream instead.
// ev (nullable): events 4 c + 2 prec and 4 c + 2 prec + 1 are recorded around each class launch;
// prim_count (nullable): 2 c + prec counts the evaluated primitive quartets of each launch.
int launch_eri_classes(hf_system* S, EriArgs a, int shard, int n_shards, int flags, cudaEvent_t* ev,
                       unsigned long long* prim_count);

// Device address of the allocation-free build's fixed scratch on the current device (noalloc.cu).
int noalloc_scratch_address(void** out);

// ---------------------------------------------------------------- errors --
struct Status {
    int code = HF_OK;
    std::string msg;
};
void set_error(int code, const std::string& msg);
int cuda_status(cudaError_t e, const char* what);

#define HF_CUDA(call)                                          \
    do {                                                       \
        cudaError_t e_ = (call);                               \
        if (e_ != cudaSuccess) return cuda_status(e_, #call);  \
    } while (0)

// -------------------------------------------------- device buffer helper --
struct DevBuf {
    void* p = nullptr;
    size_t bytes = 0;
    bool owned = true;
    int alloc(size_t n);
    void release();
    // non-owning view of part of another buffer (an arena)
    void view(void* ptr, size_t n)
    {
        release();
        p = ptr;
        bytes = n;
        owned = false;
    }
    template <typename T>
    T* as() const { return (T*)p; }
    ~DevBuf() { release(); }
    DevBuf() = default;
    DevBuf(const DevBuf&) = delete;
    DevBuf& operator=(const DevBuf&) = delete;
};

// Exponent table over the distinct primitive exponents of one or several bases (HermView::etab); empty (tab.p
// nullptr) when they give more than kHermMaxTypes sums.
struct ExponentTable {
    std::vector<double> exps;  // distinct, ascending
    DevBuf tab, psum;
    int ntype = 0;
    int build(cudaStream_t s);
    HermView view(HermView h) const
    {
        h.etab = tab.as<double2>();
        h.ntype = ntype;
        return h;
    }
};

// Adds a basis' exponents to a sorted list without repetitions.
void add_exponents(std::vector<double>& exps, const hf_basis& b);

// The context's table over these exponents: one that a live system or batch holds, or a new one (its kernel is issued
// on the context's stream, as is all work that reads it or an event that orders that work).  A table takes 1.7 MB for
// the water basis and up to 33 MB, a one-water system without it 0.3 MB: systems of one basis share it, and the last
// owner frees it.
int exponent_table(hf_ctx* ctx, std::vector<double> exps, std::shared_ptr<const ExponentTable>& out);

// Status of hf_system_create's argument checks.
int check_geometry_basis(const hf_geometry* g, const hf_basis* b, const hf_thresholds* th);

// hf_system_create on a given exponent table (nullptr: the context's over the basis' exponents), which holds every
// exponent of the basis.
int create_system(hf_ctx* ctx, const hf_geometry* geom, const hf_basis* basis, const hf_thresholds* th,
                  std::shared_ptr<const ExponentTable> table, hf_system** out);

}  // namespace hf

// hf_eigh of host arrays with the start that the SCF's diagonalisations take (EighStart::kBasis32); basis_used and sweeps
// (nullable) tell whether the basis was accepted and how many sweeps it left.  Not part of the public interface: its
// eigenvectors' signs follow the basis.
extern "C" int hf_eigh_basis32(hf_ctx* ctx, int n, const double* A, double* w, double* V, int32_t* basis_used,
                               int32_t* sweeps);

// ----------------------------------------------------------- C-ABI types --
struct hf_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    int num_sms = 0;
    hf::DevBuf boys64, boys32;  // Boys Taylor tables
    cudaEvent_t ev[4 * hf::kNumClasses + 4] = {};
    int n_systems = 0;            // live systems created on this context
    bool destroy_pending = false;  // hf_destroy was called while systems were alive
    cudaStream_t fast = nullptr;  // of higher priority: the FP32 launches beside FP64 ones
    cudaStream_t side[hf::kSideStreams] = {};  // class launches of one build run on these, forked from and
    cudaEvent_t fork = nullptr, join[hf::kSideStreams + 1] = {};  // joined to `stream` (launch_eri_classes)
    void* noalloc_scratch = nullptr;  // device address of hf_fock_build_noalloc's fixed scratch
    std::mutex tables_lock;
    std::vector<std::weak_ptr<const hf::ExponentTable>> tables;  // exponent_table: those that systems or batches hold
};

struct hf_system {
    hf_ctx* ctx = nullptr;
    int device = 0;               // copies of the context's device and stream, so that
    cudaStream_t stream = nullptr;  // destruction never needs the context
    int n_atoms = 0, n_shells = 0, n_bf = 0, n_electrons = 0;
    double E_nn = 0.0;
    hf_thresholds th{};
    // shells (device)
    hf::DevBuf sh_l, sh_atom, sh_bf0, sh_nprim, sh_prim0, sh_exp, sh_coef, atom_xyz, atom_Z;
    hf::DevBuf comp_norm;  // [n_bf] Cartesian component factor
    // pairs
    int n_pairs_all = 0, n_prim_pairs = 0;
    hf::DevBuf pairs, prims64, prims32, pair_class;
    hf::DevBuf hrec, hB;          // HermPair records and bounds (HermView)
    std::shared_ptr<const hf::ExponentTable> etab;
    hf::HermView herm{};
    int class_count[hf::kNumPairClasses] = {};
    hf::DevBuf class_ids[hf::kNumPairClasses];  // sorted significant pair ids
    double Qmax = 0.0;
    // quartet schedule per class
    struct ClassPlan {
        hf::DevBuf offsets64, offsets32, kstart32;
        hf::DevBuf chunk64, chunk32;  // bra of every 2^kChunkShift-th quartet (see EriArgs::chunk)
        long long n64 = 0, n32 = 0;
        long long n_unscreened = 0;
    } plan[hf::kNumClasses];
    // matrices (device)
    hf::DevBuf S, H, P64, P32, Jt, Kt, J, K, F, Ebuf, host_stage;
    int64_t quartets_total = 0;
    // scratch
    hf::DevBuf class_q[hf::kNumPairClasses];  // sorted bounds of class_ids
    hf::DevBuf Qall, counts, staging_P, staging_out, bad, Bprim, prim_count;
    hf::DevBuf arena_in, arena_mat, arena_sched, arena_tab;  // owners of the views above
    hf::DevBuf dsh;                                // density block maxima for density-weighted screening
    // ket tables: per pair class, the significant pairs' primitive-pair records in class-list order and
    // field-major (9 maxpp rows of FP64 fields, 9 maxpp rows of FP32 fields, maxpp rows of bounds)
    hf::DevBuf ket_tab[hf::kNumPairClasses];
    hf::DevBuf class_hdr[hf::kNumPairClasses];  // pair headers of each class list, in list order
    long long ket_stride[hf::kNumPairClasses] = {};
    int fock_copies = 1;                           // accumulator copies of Jt / Kt (1: one shared copy)
    hf::DevBuf copies;                             // [2][fock_copies][N*N] when fock_copies > 1
    int maxpp = 0;
    // host copies used by the learned guess: nuclear charges, first basis
    // function and function count of each atom (-1 if its shells are not contiguous)
    std::vector<int> Z_h, atom_bf0_h, atom_nbf_h;
};
