// Internal declarations shared by the host API and the kernel files of libisc.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "isc.h"

namespace isc {

struct TShape {
    int c, h, w;
    int cp;  // channels padded to a multiple of 16 (device NHWC layout)
};

constexpr int kNoiseGuideBits = 10, kNoiseGuide = 1 << kNoiseGuideBits;

// Table of bins, an alternative to guide and bisection.  A uniform's distance t from its nearer end of the range (u or ~u, below
// 2^31) plus 2^kNoiseBinsFrom, read as a floating-point number of `bits` bits of fraction, is its bin: bins are narrow where
// levels are, and at few bits nearly all hold at most one boundary between two levels.  Entry {boundary, level below it},
// level counted from -T, kNoiseOpen where a bin holds more.  First the bins of u, then those of ~u.
constexpr int kNoiseBinsFrom = 21, kNoiseOpen = 1 << 30;
constexpr __host__ __device__ uint32_t noise_bins_side(int bits) { return ((uint32_t)(31 - kNoiseBinsFrom) << bits) + 2u; }

// Where the random stream of one launch starts (Philox4x32-10 key and fixed counter words).
struct NoiseStream {
    uint32_t key0, key1;      // seed halves
    uint32_t ctr2;            // image_id low 32
    uint32_t ctr3_fixed;      // phase | (image_id >> 32 & 0xFFFF) << 16
    int64_t first_sample;     // sample id of batch slot 0
    const uint32_t *cum;      // device, 2T+1 entries
    int T;
    // Optional guide table (device, kNoiseGuide + 1 entries, or null): guide[j] is the search result for the
    // uniform j << (32 - kNoiseGuideBits), a lower bound of the result for every uniform with these top bits.
    const uint32_t *guide;
    int guide_steps;          // bisection steps that close the widest interval [guide[j], guide[j+1]]
    const uint2 *bins;        // device, or null
    int bin_bits;
};

// What the samples of a forward pass of the layer-by-layer kernels are: per image, n_sel samples of the selection phase (numbers
// from 0 on), then the estimation phase's (numbers from first_est on), per_image in all; a launch's samples start at number
// `first` of this sequence.  Images lie one after the other; votes go to row 2 i (selection) and 2 i + 1 (estimation) of the
// counts, or to row i without a selection phase.
struct SampleRun {
    uint64_t image_id0;
    uint64_t n_sel, per_image, first, first_est;
    uint32_t phase_sel, phase_est;
    struct Sample { uint64_t image, number; uint32_t phase, row; };
    __host__ __device__ Sample at(uint32_t slot) const
    {
        const uint64_t g = first + slot, image = g < per_image ? 0 : g / per_image, r = g - image * per_image;
        const bool sel = r < n_sel;
        return Sample{image, sel ? r : first_est + (r - n_sel), sel ? phase_sel : phase_est, (uint32_t)(n_sel ? 2 * image + (sel ? 0 : 1) : image)};
    }
};

// One layer as the layer-by-layer kernels see it (device pointers).
struct GLayer {
    int op;
    int cin, cinp, cout, coutp;
    int kh, kw, stride, pad, relu;
    int zp_in, zp_out, zp_res, res_mult, res_shift;
    int hin, win, hout, wout;
    const int8_t *w;        // conv/FC: [coutp/16][kh*kw][cinp/16][16 out][16 in]; first layer: [coutp][kh*kw][4]
    const int32_t *bias;    // [coutp], folded: bias - zp_in * sum(w)
    const int32_t *mult;    // [coutp]
    const int32_t *shift;   // [coutp]
};

// One validated layer with its host arrays, as the engines' planners receive it.
struct LayerIn {
    isc_layer d;
    const int8_t *w;
    const int32_t *bias;
    const int32_t *mult;
    const int8_t *shift;
};

// ---- layer-by-layer engine (isc_generic.cu) ----
cudaError_t launch_first_conv(const GLayer &L, const uint8_t *x_chw, int in_c, const NoiseStream &ns, const SampleRun &run,
                              int batch, int8_t *out, cudaStream_t st);
cudaError_t launch_noisy_input(const uint8_t *x_chw, int in_c, int in_h, int in_w, const NoiseStream &ns,
                               int batch, int32_t *out_chw, cudaStream_t st);
cudaError_t launch_conv(const GLayer &L, int batch, const int8_t *in, const int8_t *res, int8_t *out,
                        cudaStream_t st);
cudaError_t launch_gavgpool(const GLayer &L, int batch, const int8_t *in, int8_t *out, cudaStream_t st, bool chained = false);
cudaError_t launch_maxpool(const GLayer &L, int batch, const int8_t *in, int8_t *out, cudaStream_t st, bool chained = false);
cudaError_t launch_votes(const int8_t *logits_nhwc, int cp, int n_classes, const SampleRun &run, int batch, int32_t *counts,
                         int8_t *logits_out, cudaStream_t st, bool chained = false);

// ---- layer-by-layer tensor-core convolutions (isc_igemm.cu) ----
// What their launches need of the current device.  A handle keeps its own (calls on one handle do not overlap, so nothing
// here is shared between threads), filled by tc_prepare, which also raises the kernels' shared-memory limits there: those
// are a property of each device.
struct TcDevice {
    int ordinal = -1, n_sms = 0;
    bool chained = false;     // layers may be launched ahead of the end of the one before (see launch_chained)
    void *encode = nullptr;   // the driver's cuTensorMapEncodeTiled, or null
};
cudaError_t tc_prepare(TcDevice *dev, int ordinal);
bool igemm_takes(const GLayer &G);               // whether the implicit-GEMM kernel has a form for this layer
int igemm_tile_n(const GLayer &G);               // its output-channel tile (a multiple of 16 up to 256)
int igemm_padded_cout(const GLayer &G);          // output channels with the last tile's padding: entries of the constants
bool conv_offsets_fit(const GLayer &G, int64_t batch);  // the batch's tensors are within the tensor-core kernels' 32-bit offsets
size_t igemm_pack_bytes(const GLayer &G);
void igemm_pack_weights(const GLayer &G, const int8_t *w_oihw, int8_t *out);
// The residual term floor((u * m2 + R2) / 2^32), u = r + 128 in 0..255, of the 32-bit epilogues as a single-precision product,
// round((256 k + u) * m) - c, with round to nearest even and m one of the three single-precision numbers nearest to the
// multiplier: the smallest k < 4096 for which the two agree on all 256 inputs.  What the kernels compute where it exists (for
// more than 99 % of all multipliers), the 64-bit form otherwise.
struct ResidualForm {
    uint32_t k8 = 0xFFFFFFFFu, m_bits = 0;       // 256 k; m as stored
    bool exists() const { return k8 != 0xFFFFFFFFu; }
};
ResidualForm residual_form(int res_mult, int res_shift, int zp_res, int32_t *c);
// The 32-bit epilogues compute (hi32(acc * mult) + addend) >> s.  The loader refuses layers whose accumulators could reach
// 2^30, so the product's high word lies in [-2^29, 2^29), and this is the room that the addend has to leave it in 32 bits.
constexpr bool requant_addend_fits(long long addend) { return addend >= -(3ll << 29) && addend <= 3ll << 29; }
// Per-channel requantisation constants of the kernel's 32-bit epilogue (4 x int32 for `n_out` channels); returns
// whether the layer qualifies for it (every shift >= 2, every addend leaves room for the product).
bool igemm_constants(const GLayer &G, const int32_t *bias_folded, const int32_t *mult, const int32_t *shift, int32_t *out4, int n_out,
                     bool has_residual, ResidualForm *form);
void igemm_order_constants(const GLayer &G, int32_t *out4, int n_out);      // ... in the order in which k_igemm reads them
// `cst` / `fast`: what igemm_constants produced (device copy).  `err` (device) receives a non-zero word if a bounded
// wait inside the kernel expired.  `debug_stall`: the kernel's weights are never sent, so that its waits run out
// (after their 2 s limit) and the CTAs leave through the abort path -- nothing faults or hangs.  `tensor_copy`: a
// 1 x 1 stride-1 layer may take its operand rows by tensor copy (false: the gather warps bring them, as for every
// other layer).
cudaError_t launch_igemm_conv(const TcDevice &dev, const GLayer &G, const int8_t *wpack, const int32_t *cst, bool fast, const ResidualForm &form, int batch, const int8_t *in,
                              const int8_t *res, int8_t *out, int32_t *err, cudaStream_t st, bool debug_stall = false,
                              bool tensor_copy = true);

// ---- stride-1 "same" convolutions with the input tile in shared memory (isc_halo.cu) ----
// Odd square filters from 3 x 3 on whose tile fits.  Constants as igemm_constants makes them, for halo_padded_cout channels.
bool halo_fits(const GLayer &G);
bool halo_offsets_fit(const GLayer &G, int64_t batch);
int halo_padded_cout(const GLayer &G);
size_t halo_pack_bytes(const GLayer &G);
void halo_pack(const GLayer &G, const int8_t *w_oihw, int8_t *out);
void halo_order_constants(const GLayer &G, int32_t *out4, int n_out);      // igemm_constants' in the order in which k_halo reads them
cudaError_t halo_prepare();                      // part of tc_prepare
cudaError_t launch_halo_conv(const TcDevice &dev, const GLayer &G, const int8_t *wpack, const int32_t *cst, bool fast, const ResidualForm &form, int batch,
                             const int8_t *in, const int8_t *res, int8_t *out, int32_t *err, cudaStream_t st, bool debug_stall = false);

// The first convolution (<= 4 input channels, filter at most 8 x 8) on the tensor cores, noise drawn into its staging.
bool stem_fits(const GLayer &G, int in_c);
size_t stem_pack_bytes(const GLayer &G);
void stem_pack_weights(const GLayer &G, const int8_t *w_oihw, int8_t *out);
cudaError_t launch_stem_conv(const TcDevice &dev, const GLayer &G, const int8_t *wpack, const int32_t *cst, bool fast, const uint8_t *x_chw, int in_c,
                             const NoiseStream &ns, const SampleRun &run, int batch, int8_t *out, int32_t *err, cudaStream_t st, bool debug_stall = false,
                             bool chained = false);

// ---- host decision rules (isc_decide.cpp) ----
double lower_conf_bound(int64_t k, int64_t n, double alpha);
double normal_quantile(double p);
double binom_pvalue_half(int64_t n_a, int64_t m);
int32_t decide_certify(const int32_t *counts0, const int32_t *counts, int n_classes, int64_t N,
                       double sigma, double alpha, double *radius, double *p_lower);
int32_t decide_predict(const int32_t *counts, int n_classes, double alpha);
// `table`: Eq. 2's cumulative table for sigma (n_table entries) if the caller has it, else null
int32_t decide_certify_integer(const int32_t *counts0, const int32_t *counts, int n_classes, int64_t N, double sigma,
                               double alpha, bool two_sided, int32_t *q, int64_t *q_squared, const uint32_t *table, size_t n_table);
int noise_halfwidth(double sigma);
void noise_table(double sigma, std::vector<uint32_t> &cum);
void noise_table_rounded(double sigma, std::vector<uint32_t> &cum);

}  // namespace isc
