// nb_ext.h -- services of the context (nb_capi.cu) used by the translation
// units that implement the other entry points (leap-frog, batched, VJP).
#pragma once

#include <cstdint>
#include <string>

#include "nb_internal.h"

namespace nbx {

// Grow-only device buffers owned by the context for the other entry points,
// one per slot id (every translation unit takes its ids from this list).
enum ExtSlot : int {
    SLOT_FP64_JP = 0,   // packed particles from FP64 state (leap-frog, energy)
    SLOT_ENERGY_A,      // accelerations computed by nb_energy
    SLOT_P,             // potentials computed by nb_energy
    SLOT_ENERGY_BLK,    // energy block sums
    SLOT_ENERGY_OUT,    // energy result
    SLOT_BATCH_PLAN,    // batched: what the plan was made for, offsets and blocks
    SLOT_BATCH_ITEMS,   // batched: work items
    SLOT_VJP_VP,        // packed VJP records
    SLOT_VJP_PART,      // VJP partial sums
    SLOT_HL_BOX,        // bounding-box partials of FP64 positions (HL packing)
    SLOT_ADJOINT,       // leap-frog adjoint: replayed state, position history, VJP operands
    SLOT_BATCH_FRAME,   // per-cluster HL frames (centre, grid) of the batched leap-frog
    SLOT_BATCH_CP,      // batched: packed particles
    SLOT_BATCH_PI,      //   sums of the i-side
    SLOT_BATCH_PJ,      //   sums of the j-side
    SLOT_MUTUAL_NOTES,  // mutual kernels: the form of the weights, and what the pack found
    SLOT_MUTUAL,        //   the other scratch of each user (mutual_slot)
    SLOT_COUNT = SLOT_MUTUAL + 15
};

// The calls that run mutual kernels, each with scratch of its own: a captured nb_force
// must find its buffers where they were, whatever the other calls need meanwhile.
enum MutualUser : int { kMutualForce = 0, kMutualFp64 = 1, kMutualVjp = 2 };
enum MutualPart : int {
    kPartCp = 0,  // packed particles
    kPartPi,      // segment sums of the i-side
    kPartPj,      // j-side sums of a panel of rows
    kPartRows,    // first and last CTA of each row
    kPartState,   // sums carried from panel to panel
    kMutualParts
};
inline int mutual_slot(MutualUser user, MutualPart part) { return SLOT_MUTUAL + kMutualParts * user + part; }
static_assert(SLOT_COUNT == SLOT_MUTUAL + 3 * kMutualParts, "every part of every user");

struct ExtState {
    static constexpr int kSlots = SLOT_COUNT;
    void *buf[kSlots] = {};
    size_t cap[kSlots] = {};
    int vjp_idx = -1;  // VJP shape forced by nb_set_vjp_tile (-1: built-in)
    // Largest n whose mutual scratch is known not to have failed to allocate:
    // above it the built-in choice is a direct shape.
    int64_t mutual_max_n = INT64_MAX, vjp_mutual_max_n = INT64_MAX;
    int64_t batch_max_n = INT64_MAX;  // (padded particles; above it: the small scratch)
    bool batch_plan = false;          // a plan was launched into SLOT_BATCH_PLAN
};
void ext_release(ExtState &s);

// Brackets one kernel launch (or `launches` of them) with CUDA events on its
// stream when the context's timing is on (nb_timing_enable).
class TimedLaunch {
  public:
    TimedLaunch(nb_ctx *ctx, int kernel, cudaStream_t st, int launches = 1);
    ~TimedLaunch();
    TimedLaunch(const TimedLaunch &) = delete;
    TimedLaunch &operator=(const TimedLaunch &) = delete;

  private:
    nb_ctx *ctx_;
    int kernel_;
    int launches_;
    cudaStream_t st_;
    cudaEvent_t start_ = nullptr, stop_ = nullptr;
};

nb_status fail(nb_ctx *ctx, nb_status st, const std::string &m);
// Message returned by nb_last_error(NULL) (calls without a context).
void set_global_error(const std::string &m);
nb_status cuda_fail(nb_ctx *ctx, cudaError_t e, const char *what);
nb_status check_common(nb_ctx *ctx, int64_t n, float eps, int mode);

int ctx_device(const nb_ctx *ctx);
int ctx_sm_count(const nb_ctx *ctx);
int *ctx_err_word(nb_ctx *ctx);
uint64_t ctx_wait_ns(const nb_ctx *ctx);
int64_t ctx_fault_unit(const nb_ctx *ctx);
ExtState &ctx_ext(nb_ctx *ctx);
// Turn per-kernel event timing on or off; returns the previous setting.
bool ctx_set_timing(nb_ctx *ctx, bool on);

cudaError_t ensure_buffer(void **ptr, size_t *cap, size_t bytes);
// CTAs of the kernel on the GPU at once. `most`: the most dynamic shared memory that a
// launch of it asks for, where that is more than v.smem; the same for every context,
// because the limit it sets on the kernel is the process's.
int resident_ctas(nb_ctx *ctx, const nbk::PairVariant &v, size_t most = 0);
const nbk::PairVariant &choose_variant(nb_ctx *ctx, int64_t n, bool comp);

// Compensated path on FP64 state: pair kernel on HL records (two JParts per
// particle, nbk::kHLRecords), then the compensated combine; p may be NULL
// (the potential is then not summed). only_p: a is zeroed, not summed.
nb_status run_force_hl(nb_ctx *ctx, const nbk::JPart *jp, int64_t n, float eps, float *a, float *p,
                       cudaStream_t st, bool only_p = false);
// Allocate what the direct shapes need for n, whichever is picked.
nb_status reserve_direct(nb_ctx *ctx, int64_t n, bool comp);
// Allocate the HL path's partial sums for n (before any graph capture).
nb_status reserve_hl(nb_ctx *ctx, int64_t n);

// pack (unless prepacked) -> pair -> combine, enqueued on st.
nb_status run_force(nb_ctx *ctx, const float *x, const float *m, const nbk::JPart *prepacked,
                    int64_t n, float eps, float *a, float *p, bool comp, cudaStream_t st,
                    bool only_p = false);

// Mutual kernels (nb_mutual.cu). mutual_reserve allocates what n needs; the
// records are then packed by run_mutual from x, m, or, with x NULL (the calls on FP64
// state, kMutualFp64), by a kernel of the caller's (mutual_pack_blocks blocks of kMutualPackThreads) into
// mutual_records, with mutual_note on mutual_notes. a or p may be NULL.
constexpr int kMutualPackThreads = 128;
inline int64_t mutual_pack_blocks(int64_t npad) { return (npad + kMutualPackThreads - 1) / kMutualPackThreads; }
// The index of the mutual shape that a call on n FP64 positions takes, or -1:
// the built-in one, or for a plain call the one forced or tuned.
int mutual_from_fp64(nb_ctx *ctx, int64_t n, bool comp);
int64_t mutual_npad(const nbk::MutualShape &s, int64_t n);
nb_status mutual_reserve(nb_ctx *ctx, const nbk::MutualShape &s, int64_t n, MutualUser user);
float4 *mutual_records(nb_ctx *ctx, MutualUser user);
int *mutual_notes(nb_ctx *ctx);
nb_status run_mutual(nb_ctx *ctx, const nbk::MutualShape &s, const float *x, const float *m, int64_t n, float eps,
                     float *a, float *p, cudaStream_t st);

// A step of the leap-frog's adjoint around its VJP of Eq. (gravity), all FP64: the
// operands are x and la with the back kick's share -dt/2 lv (first: the force at the
// start of a trajectory, la alone), and the result enters lx and lm, then the drift
// and the front kick lv and la (first: la is cleared).
struct VjpState {
    const double *x;
    double *lx, *lv, *la, *lm;
    double dt;
    int first;
};

// nb_force_vjp on the mutual kernels (nb_vjp_mutual.cu); gp may be NULL. With a
// state: from and to its arrays, not x, ga, gp, gx, gm. NB_ERR_OOM when the scratch
// cannot be allocated (nothing is enqueued then).
nb_status run_vjp_mutual(nb_ctx *ctx, int size, const float *x, const float *m, int64_t n, float eps, const float *ga,
                         const float *gp, float *gx, float *gm, cudaStream_t st, const VjpState *state = nullptr);
// The size argument for n without an upstream gradient on p, -1 for a direct shape.
int vjp_mutual_size(nb_ctx *ctx, int64_t n);

struct DeviceGuard {
    int prev = -1;
    bool changed = false;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) changed = cudaSetDevice(dev) == cudaSuccess;
    }
    ~DeviceGuard() {
        if (changed) cudaSetDevice(prev);
    }
};

}  // namespace nbx
