// Forward-table kernels and their launch plumbing (internal to libgbs).
#pragma once
#include <cstddef>
#include <cstdint>
#include <string>
#include <cuda_runtime.h>

namespace gbs {

// Table a forward call fills: vacuum probabilities, click moments, click
// cumulants, spin correlators c(S) (Eq. correlator_sum_cov), spin cumulants
// kappa(S) (Eq. cumulant_corr_main).
enum Mode : int { MODE_P0 = 0, MODE_MU = 1, MODE_KAPPA = 2, MODE_SPINC = 3, MODE_SPINK = 4 };

// Everything one forward call needs on the device. Tables use the layout of
// gbs.h (order groups, colex ranks within an order).
struct FwdArgs {
    const double *V;      // 2M x 2M covariance (row-major, xxpp)
    const double *mean;   // first moments (2M, xxpp) of a displaced state; nullptr = zero mean
    int M, kmax, mode, precision;
    double *A;            // packed 2x2 blocks of (V+I)/2, M*M*4 doubles (workspace)
    float *Af;            // the same blocks as float pairs (hi x4, lo x4), refined path (workspace)
    // refined cumulant calls with kmax >= 4: the lower orders' P0 and no-click cumulants
    // ky (gbs_tree.cuh, combine_products) as float pairs (workspace; null otherwise)
    float2 *p0p, *kyp;
    double *p0;           // P0 table: the output for MODE_P0, a workspace table (orders < kmax) otherwise
    double *out;          // mu or kappa table (MODE_MU / MODE_KAPPA); equals p0 for MODE_P0
    unsigned *status;     // status word (workspace)
    unsigned *counters;   // per-order work counters (workspace, zeroed per call)
    double *scratch;      // per-CTA Schur-complement slots (workspace)
    size_t slot_doubles;  // doubles per slot
    int slots;            // number of slots = max persistent CTAs
    int sms;              // multiprocessors on the device
    cudaEvent_t *ev;      // GBS_MAX_ORDER + 2 timing events, or nullptr
    // range call (gbs_table_range): order kmax is filled only for top elements in
    // [c_lo, c_hi), into top[idx - top_base]; top = nullptr fills whole tables
    double *top;
    uint64_t top_base;
    int c_lo, c_hi;
    // prefix-tree schedule (autotuned): items per CTA slot, children per shared-
    // memory batch, CTA shape (0: 512 threads x 1 per SM; 1: 256 x 2; 4: 256 x 3 with a
    // 672-entry x area; refined path only: 2: 128 x 6 with a 304-entry x area, 3: 256 x
    // 3, 5: 384 x 2 with a 960-entry x area, 6: 256 x 4 with a 384-entry x area, 7: 6 in
    // clusters of 4, 8: 3 in clusters of 3, 9: 6 without Schur-complement slots)
    int grain, ccap, variant;
};

// Valid (M, kmax) of a forward table: orders 4 and 5 run the prefix-tree kernels
// (shared-memory x-entries sized for GBS_MAX_MODES); tables with kmax <= 3 run
// order 3 by chunks and take up to GBS_MAX_MODES_K3 modes.
inline bool valid_mk(int M, int kmax) {
    return M >= 1 && kmax >= 1 && kmax <= 5 && kmax <= M && M <= (kmax <= 3 ? 4096 : 1024);
}

// Message for an (M, kmax) that valid_mk rejects (defined in gbs_api.cu).
std::string shape_message(int M, int kmax);

// Schedule of the prefix-tree kernels for one problem shape.
struct TreeCfg {
    int grain, ccap, variant;
};
constexpr TreeCfg kDefaultCfg{2, 64, 0};
// Most children per shared-memory batch any CTA shape has room for.
constexpr int kMaxChildren = 64;
// Largest M the 256-thread variant accepts (its shared x-entry area holds 576 modes).
constexpr int kVariant1MaxM = 577;
// x-entries per batch of the 128-thread x 6 refined variant (24 children), and its
// largest M.
constexpr int kSmallXC = 304;
constexpr int kVariant2MaxM = kSmallXC + 1;
// x-entries per batch of the second 256-thread x 3 refined variant (24 children).
constexpr int kWideXC = 672;
constexpr int kVariant4MaxM = kWideXC + 1;
// x-entries per batch of the 384-thread x 2 refined variant, and its largest M.
constexpr int kPairXC = 960;
constexpr int kVariant5MaxM = kPairXC + 1;
// x-entries per batch of the 256-thread x 4 refined variant, and its largest M.
constexpr int kQuadXC = 384;
constexpr int kVariant6MaxM = kQuadXC + 1;
// Children per batch the shapes with small or wide x areas have room for. The
// slot-free 256-thread x 4 refined variant: the elimination rows Y(x), x < c4 <= M - 2,
// it keeps in shared memory.
constexpr int kNoSlotCC = 24;
constexpr int kNoSlotYC = 160;
constexpr int kVariant9MaxM = kNoSlotYC + 1;  // order 4 reaches c4 = M - 1
// Schedule of an untuned forward call, from sweeps of shape x grain (kt, M = 20 to
// 300, kmax = 4 and 5; the tuner still finds the last percents):
//   refined, kmax = 5: 128 x 6 where its x area admits M (M = 144: 10.76 ms against
//     10.81 at 256 x 3 and 14.3 at 512 x 1; M = 77: 0.64 against 0.66 and 1.05), one
//     item per CTA slot below 128 modes, where a second round of items would wait
//     for the first, else two; kmax = 4: 256 x 3, two items (M = 144: 0.44 against
//     0.50 at 128 x 6), but 256 x 4 for the tables without gathers on pairs (P0, M =
//     100, kmax = 4: 124 us the call against 140); larger M
//     256 x 3, then 384 x 2;
//   FP64: the wide 256 x 3, one item per CTA slot (M = 111, kmax = 5: 10.9 against
//     11.2 at 256 x 2 and 12.3 at 512 x 1; M = 50: 0.32 against 0.34 and 0.47); a
//     kmax = 4 table large enough for the prefix tree (gbs_launch.cuh) 512 x 1 with
//     eight (M = 300: 23.5 against 24.9).
inline TreeCfg default_cfg(int M, int kmax, int precision, int mode) {
    TreeCfg c = kDefaultCfg;
    if (precision == 1) {
        const bool cumulants = mode == MODE_KAPPA || mode == MODE_SPINK;
        c.variant = kmax == 5 && M <= kVariant2MaxM                ? 2
                    : kmax == 4 && !cumulants && M <= kVariant6MaxM ? 6
                    : M <= kVariant4MaxM                            ? 4
                    : M <= kVariant5MaxM                            ? 5
                                                                    : 0;
        c.grain = kmax == 5 && M < 128 ? 1 : 2;
    } else if (kmax == 5) {
        c.variant = M <= kVariant4MaxM ? 4 : 0;
        c.grain = c.variant == 4 ? 1 : 2;
    } else {
        c.grain = 8;
    }
    return c;
}
// Number of CTA shapes (variants 0..kNumVariants-1); 7 and 8 are the 256 x 4 and
// 256 x 3 shapes in thread-block clusters of 4 and 3 CTAs sharing one slot, 9 the
// 256 x 4 shape without slots.
constexpr int kNumVariants = 10;
// CTA shape a forward call of (M, precision) runs for a recorded variant: the
// shapes that do not admit M (or the precision) fall back to 512 x 1.
inline int effective_variant(int variant, int M, int precision) {
    if (variant == 1 || variant == 3 || variant == 8) return M <= kVariant1MaxM && (variant == 1 || precision == 1) ? variant : 0;
    if (variant == 4) return M <= kVariant4MaxM ? 4 : 0;
    if (precision != 1) return 0;
    if (variant == 2) return M <= kVariant2MaxM ? 2 : 0;
    if (variant == 5) return M <= kVariant5MaxM ? 5 : 0;
    if (variant == 6 || variant == 7) return M <= kVariant6MaxM ? variant : 0;
    if (variant == 9) return M <= kVariant9MaxM ? 9 : 0;
    return 0;
}
// Whether a variant runs in clusters (the batched kernel has no clustered form).
inline bool variant_clustered(int v) { return v == 7 || v == 8; }

// Workspace layout, shared by the size query and the launcher.
struct WsLayout {
    size_t status_off, A_off, p0_off, scratch_off, p0p_off, kyp_off, total;
    size_t slot_doubles;
    int slots;
};
// Scratch slots per multiprocessor that cover every CTA shape allowed for M:
// six when the 128 x 6 shape can run (M <= 305), four for 256 x 4 (M <= 385), else
// three.
inline int slots_per_sm_for(int M) { return M <= kVariant2MaxM ? 6 : M <= kVariant6MaxM ? 4 : 3; }
// Reserves slots_per_sm scratch slots per multiprocessor (0 = slots_per_sm_for(M);
// with one, only one CTA per multiprocessor runs).
// pairs: with the float-pair tables of refined cumulant calls (kmax >= 4).
WsLayout ws_layout(int M, int kmax, int sms, int slots_per_sm, bool pairs);

// Queues every kernel of one forward call on stream; returns a cudaError_t.
cudaError_t launch_forward(const FwdArgs &a, cudaStream_t stream);
// The same for a displaced state (a.mean set, a.precision = 0).
cudaError_t launch_forward_displaced(const FwdArgs &a, cudaStream_t stream);

}  // namespace gbs
