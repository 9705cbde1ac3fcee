// Host side of libisc: argument checks, model repacking and upload, launch sequencing of the
// Monte-Carlo loop (Algorithm 1 steps 1-4, Algorithm 2 steps 1-2) and the decision rules.
#include <cuda_runtime.h>

#include <chrono>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "isc.h"
#include "isc_internal.h"
#include "isc_line.h"

using namespace isc;

namespace {

inline int pad16(int c) { return (c + 15) & ~15; }

struct HostLayer {           // private copy of one isc_layer with its arrays
    isc_layer d;
    std::vector<int8_t> w;
    std::vector<int32_t> bias, mult;
    std::vector<int8_t> shift;
};

struct DevBuf {
    void *p = nullptr;
    size_t bytes = 0;
};

}  // namespace

struct isc_model {
    int in_c = 0, in_h = 0, in_w = 0, n_classes = 0;
    std::vector<HostLayer> layers;
    std::vector<TShape> shapes;                 // [n_layers + 1]
    int64_t macs = 0;

    // device parameters of the layer-by-layer engine
    std::vector<GLayer> glayers;
    std::vector<void *> param_allocs;
    std::vector<const int8_t *> wpacks;         // per layer: weights repacked for k_igemm (layer 0: k_stem), or null
    std::vector<const int8_t *> hpacks;         // per layer: weights repacked for k_halo, which takes the layer then, or null
    std::vector<const int32_t *> tc_cst;        // per layer: its epilogue constants
    std::vector<char> tc_fast;
    std::vector<isc::ResidualForm> tc_resk;  // per layer: the residual term as a single-precision product, where that exists
    bool has_tc = false;
    isc::TcDevice tc;
    int32_t *d_tc_err = nullptr;                // error word of the stalled launches (see stalled_launch)

    // activation buffers: tensor t lives in pool buffer tensor_buf[t] (bytes per sample buf_bytes[b])
    std::vector<int> tensor_buf;
    std::vector<size_t> buf_bytes;
    std::vector<DevBuf> bufs;
    int ws_batch = 0;
    int64_t ws_limit = INT64_MAX;               // samples that the device's memory held when it did not hold more

    // per-call device scratch
    // One buffer: error word (16 bytes), vote counts, images.  A call's upload (zeros and images) and its download (error
    // word and counts) are one copy each, through the pinned buffer, whose front both share.
    uint8_t *d_io = nullptr;      size_t d_io_bytes = 0;
    uint8_t *h_io = nullptr;      size_t h_io_bytes = 0;
    int8_t *d_logits = nullptr;   size_t d_logits_bytes = 0;
    uint32_t *d_cum = nullptr;    size_t d_cum_n = 0;
    double cum_sigma = -1.0;                    // what d_cum holds
    int cum_kind = -1;
    // the table on the host: the cumulative one, the guide, the bins if the law has them
    std::vector<uint32_t> h_tab;
    double tab_sigma = -1.0;
    int tab_T = 0, tab_kind = -1, tab_steps = 0, tab_bin_bits = 0;
    size_t tab_front = 0;                       // entries before the bins

    isc::LinePlan *line = nullptr;

    // isc_certify_batch: one event per piece of the batch
    std::vector<cudaEvent_t> events;

    int64_t opt_batch = 0, opt_engine = 0, opt_noise = 0, opt_tensor_copy = 1;
    int64_t last_engine = 0, last_static_engine = 0, launches = 0;
};

namespace {

#define CK(call)                                      \
    do {                                              \
        cudaError_t e_ = (call);                      \
        if (e_ != cudaSuccess) {                      \
            if (getenv("ISC_DEBUG_CUDA")) fprintf(stderr, "isc: %s: %s\n", #call, cudaGetErrorString(e_)); \
            cudaGetLastError();                       \
            return e_ == cudaErrorMemoryAllocation ? ISC_ERR_NOMEM : ISC_ERR_CUDA; \
        }                                             \
    } while (0)

int infer_shape(const isc_layer &L, const TShape &in, TShape *out)
{
    switch (L.op) {
    case ISC_CONV2D:
    case ISC_MAXPOOL:
        if (L.kh < 1 || L.kw < 1 || L.stride < 1 || L.pad < 0) return ISC_ERR_SHAPE;
        if (L.cin != in.c) return ISC_ERR_SHAPE;
        if (in.h + 2 * L.pad < L.kh || in.w + 2 * L.pad < L.kw) return ISC_ERR_SHAPE;
        if (L.op == ISC_MAXPOOL && L.cout != L.cin) return ISC_ERR_SHAPE;
        if (L.cout < 1) return ISC_ERR_SHAPE;
        out->c = L.cout;
        out->h = (in.h + 2 * L.pad - L.kh) / L.stride + 1;
        out->w = (in.w + 2 * L.pad - L.kw) / L.stride + 1;
        break;
    case ISC_FC:
        if (in.h != 1 || in.w != 1 || L.cin != in.c || L.cout < 1) return ISC_ERR_SHAPE;
        out->c = L.cout; out->h = 1; out->w = 1;
        break;
    case ISC_GAVGPOOL:
        if (L.cin != in.c || L.cout != in.c) return ISC_ERR_SHAPE;
        out->c = in.c; out->h = 1; out->w = 1;
        break;
    default:
        return ISC_ERR_ARG;
    }
    out->cp = pad16(out->c);
    return ISC_OK;
}

template <typename T>
int upload(isc_model *m, const std::vector<T> &h, const T **dptr)
{
    void *p = nullptr;
    CK(cudaMalloc(&p, std::max<size_t>(h.size() * sizeof(T), 16)));
    m->param_allocs.push_back(p);
    CK(cudaMemcpy(p, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice));
    *dptr = static_cast<const T *>(p);
    return ISC_OK;
}

// Validate, copy, infer shapes.  No device work.
int build_host_model(isc_model *m, const isc_layer *layers, int n_layers)
{
    m->shapes.resize((size_t)n_layers + 1);
    m->shapes[0] = TShape{m->in_c, m->in_h, m->in_w, 4};
    m->layers.resize((size_t)n_layers);
    std::vector<int> uses_of_input(1, 0);
    for (int i = 0; i < n_layers; ++i) {
        const isc_layer &L = layers[i];
        if (L.op < ISC_CONV2D || L.op > ISC_MAXPOOL) return ISC_ERR_ARG;
        if (L.in_tensor < 0 || L.in_tensor > i) return ISC_ERR_SHAPE;
        if (L.res_tensor < -1 || L.res_tensor > i) return ISC_ERR_SHAPE;
        const bool weighted = L.op == ISC_CONV2D || L.op == ISC_FC;
        if (L.res_tensor >= 0 && !weighted) return ISC_ERR_SHAPE;
        if (!L.mult || !L.shift) return ISC_ERR_ARG;
        if (weighted && (!L.w || !L.bias)) return ISC_ERR_ARG;
        int rc = infer_shape(L, m->shapes[(size_t)L.in_tensor], &m->shapes[(size_t)i + 1]);
        if (rc) return rc;
        const TShape &os = m->shapes[(size_t)i + 1];
        if (L.res_tensor >= 0) {
            const TShape &r = m->shapes[(size_t)L.res_tensor];
            if (L.res_tensor == 0 || r.c != os.c || r.h != os.h || r.w != os.w) return ISC_ERR_SHAPE;
            if (L.res_mult < (1 << 30) || L.res_shift < -4 || L.res_shift > 4) return ISC_ERR_ARG;
            if (L.zp_res < -128 || L.zp_res > 127) return ISC_ERR_ARG;
        }
        const int zp_in_lo = L.in_tensor == 0 ? 0 : -128, zp_in_hi = L.in_tensor == 0 ? 255 : 127;
        if (L.zp_in < zp_in_lo || L.zp_in > zp_in_hi) return ISC_ERR_ARG;
        if (L.zp_out < -128 || L.zp_out > 127) return ISC_ERR_ARG;
        if (L.relu != 0 && L.relu != 1) return ISC_ERR_ARG;

        HostLayer &H = m->layers[(size_t)i];
        H.d = L;
        const int nch = weighted ? L.cout : 1;
        H.mult.assign(L.mult, L.mult + nch);
        H.shift.assign(L.shift, L.shift + nch);
        for (int c = 0; c < nch; ++c) {
            if (L.op != ISC_MAXPOOL && H.mult[(size_t)c] < (1 << 30)) return ISC_ERR_ARG;
            if (H.shift[(size_t)c] < 0 || H.shift[(size_t)c] > 31) return ISC_ERR_ARG;
        }
        if (weighted) {
            const int kh = L.op == ISC_FC ? 1 : L.kh, kw = L.op == ISC_FC ? 1 : L.kw;
            const size_t per_out = (size_t)L.cin * kh * kw;
            H.w.assign(L.w, L.w + per_out * L.cout);
            H.bias.assign(L.bias, L.bias + L.cout);
            H.d.kh = kh; H.d.kw = kw;
            if (L.op == ISC_FC) { H.d.stride = 1; H.d.pad = 0; }
            // worst-case accumulator magnitude must stay inside int32
            const int amax = 255;                              // |a - zp_in| <= 255 for 8-bit activations
            for (int o = 0; o < L.cout; ++o) {
                int64_t s = 0;
                for (size_t k = 0; k < per_out; ++k) {
                    const int wv = H.w[(size_t)o * per_out + k];
                    if (wv == -128) return ISC_ERR_ARG;        // symmetric int8 weights: [-127, 127]
                    s += std::abs(wv);
                }
                const int64_t b = H.bias[(size_t)o];
                if (s * amax + (b < 0 ? -b : b) >= (1ll << 30)) return ISC_ERR_UNSUPPORTED;
            }
            m->macs += (int64_t)os.h * os.w * L.cout * (int64_t)per_out;
        }
        H.d.w = nullptr; H.d.bias = nullptr; H.d.mult = nullptr; H.d.shift = nullptr;
    }
    const TShape &last = m->shapes[(size_t)n_layers];
    if (last.c != m->n_classes || last.h != 1 || last.w != 1) return ISC_ERR_SHAPE;
    return ISC_OK;
}

// Device parameters and buffer plan of the layer-by-layer engine.
int build_generic_engine(isc_model *m)
{
    const int n = (int)m->layers.size();
    // tensor 0 exists only inside the first convolution's staging
    const isc_layer &L0 = m->layers[0].d;
    if (L0.op != ISC_CONV2D || L0.in_tensor != 0 || L0.cin > 4) return ISC_ERR_UNSUPPORTED;
    for (int i = 1; i < n; ++i)
        if (m->layers[(size_t)i].d.in_tensor == 0) return ISC_ERR_UNSUPPORTED;

    m->glayers.resize((size_t)n);
    m->wpacks.assign((size_t)n, nullptr);
    m->tc_cst.assign((size_t)n, nullptr);
    m->hpacks.assign((size_t)n, nullptr);
    m->tc_fast.assign((size_t)n, 0);
    m->tc_resk.assign((size_t)n, isc::ResidualForm());
    for (int i = 0; i < n; ++i) {
        const HostLayer &H = m->layers[(size_t)i];
        const isc_layer &L = H.d;
        const TShape &is = m->shapes[(size_t)L.in_tensor], &os = m->shapes[(size_t)i + 1];
        GLayer G;
        memset(&G, 0, sizeof(G));
        G.op = L.op;
        G.cin = L.cin; G.cinp = i == 0 ? 4 : is.cp;
        G.cout = L.cout; G.coutp = os.cp;
        G.kh = L.kh; G.kw = L.kw; G.stride = L.stride; G.pad = L.pad; G.relu = L.relu;
        G.zp_in = L.zp_in; G.zp_out = L.zp_out; G.zp_res = L.zp_res;
        G.res_mult = L.res_mult; G.res_shift = L.res_shift;
        G.hin = is.h; G.win = is.w; G.hout = os.h; G.wout = os.w;
        const bool weighted = L.op == ISC_CONV2D || L.op == ISC_FC;
        std::vector<int32_t> mult((size_t)(weighted ? G.coutp : 1), 1 << 30), shift(mult.size(), 0);
        for (size_t c = 0; c < H.mult.size(); ++c) { mult[c] = H.mult[c]; shift[c] = H.shift[c]; }
        int rc = upload(m, mult, &G.mult); if (rc) return rc;
        rc = upload(m, shift, &G.shift); if (rc) return rc;
        if (weighted) {
            const int taps = L.kh * L.kw;
            std::vector<int32_t> bias((size_t)G.coutp, 0);
            for (int o = 0; o < L.cout; ++o) {
                int64_t s = 0;
                for (int k = 0; k < L.cin * taps; ++k) s += H.w[(size_t)o * L.cin * taps + k];
                bias[(size_t)o] = (int32_t)(H.bias[(size_t)o] - (int64_t)L.zp_in * s);   // padding value is zp_in
            }
            rc = upload(m, bias, &G.bias); if (rc) return rc;
            std::vector<int8_t> w;
            if (i == 0) {                                   // [coutp][taps][4]
                w.assign((size_t)G.coutp * taps * 4, 0);
                for (int o = 0; o < L.cout; ++o)
                    for (int c = 0; c < L.cin; ++c)
                        for (int t = 0; t < taps; ++t)
                            w[((size_t)o * taps + t) * 4 + c] = H.w[((size_t)o * L.cin + c) * taps + t];
            } else {                                        // [coutp/16][taps][cinp/16][16 out][16 in]
                const int c16s = G.cinp / 16;
                w.assign((size_t)G.coutp * taps * G.cinp, 0);
                for (int o = 0; o < L.cout; ++o)
                    for (int c = 0; c < L.cin; ++c)
                        for (int t = 0; t < taps; ++t) {
                            const size_t idx = ((((size_t)(o / 16) * taps + t) * c16s + c / 16) * 16 + o % 16) * 16 + c % 16;
                            w[idx] = H.w[((size_t)o * L.cin + c) * taps + t];
                        }
            }
            rc = upload(m, w, &G.w); if (rc) return rc;
            if (i == 0 && stem_fits(G, m->in_c)) {          // the stem for the tensor-core kernel
                std::vector<int8_t> wp(stem_pack_bytes(G));
                stem_pack_weights(G, H.w.data(), wp.data());
                rc = upload(m, wp, &m->wpacks[0]); if (rc) return rc;
                std::vector<int32_t> c4((size_t)igemm_padded_cout(G) * 4);
                m->tc_fast[0] = igemm_constants(G, bias.data(), mult.data(), shift.data(), c4.data(), igemm_padded_cout(G), false, nullptr) ? 1 : 0;
                rc = upload(m, c4, &m->tc_cst[0]); if (rc) return rc;
            }
            const bool halo = i > 0 && halo_fits(G);
            if (halo || (i > 0 && igemm_takes(G))) {        // the same layer for the tensor-core kernel that takes it
                std::vector<int8_t> wp(halo ? halo_pack_bytes(G) : igemm_pack_bytes(G));
                if (halo) halo_pack(G, H.w.data(), wp.data()); else igemm_pack_weights(G, H.w.data(), wp.data());
                rc = upload(m, wp, halo ? &m->hpacks[(size_t)i] : &m->wpacks[(size_t)i]); if (rc) return rc;
                const int n_cst = halo ? halo_padded_cout(G) : igemm_padded_cout(G);
                std::vector<int32_t> c4((size_t)n_cst * 4);
                m->tc_fast[(size_t)i] = igemm_constants(G, bias.data(), mult.data(), shift.data(), c4.data(), n_cst, H.d.res_tensor >= 0, &m->tc_resk[(size_t)i]) ? 1 : 0;
                if (halo) halo_order_constants(G, c4.data(), n_cst); else igemm_order_constants(G, c4.data(), n_cst);
                rc = upload(m, c4, &m->tc_cst[(size_t)i]); if (rc) return rc;
                m->has_tc = true;
            }
        }
        m->glayers[(size_t)i] = G;
    }
    // buffer plan: greedy reuse by last use
    std::vector<int> last_use((size_t)n + 1, -1);
    for (int i = 0; i < n; ++i) {
        last_use[(size_t)m->layers[(size_t)i].d.in_tensor] = i;
        if (m->layers[(size_t)i].d.res_tensor >= 0) last_use[(size_t)m->layers[(size_t)i].d.res_tensor] = i;
    }
    last_use[(size_t)n] = n;
    m->tensor_buf.assign((size_t)n + 1, -1);
    std::vector<int> owner;                                 // pool buffer -> tensor currently in it (or -1)
    for (int i = 0; i < n; ++i) {
        const int t = i + 1;
        const TShape &s = m->shapes[(size_t)t];
        const size_t need = (size_t)s.h * s.w * s.cp;
        for (size_t b = 0; b < owner.size(); ++b)           // release buffers whose tensor is dead
            if (owner[b] >= 0 && last_use[(size_t)owner[b]] < i) owner[b] = -1;
        int pick = -1;
        for (size_t b = 0; b < owner.size(); ++b)
            if (owner[b] < 0 && (pick < 0 || m->buf_bytes[b] > m->buf_bytes[(size_t)pick])) pick = (int)b;
        if (pick < 0) {
            owner.push_back(-1);
            m->buf_bytes.push_back(0);
            pick = (int)owner.size() - 1;
        }
        m->buf_bytes[(size_t)pick] = std::max(m->buf_bytes[(size_t)pick], need);
        owner[(size_t)pick] = t;
        m->tensor_buf[(size_t)t] = pick;
    }
    m->bufs.resize(owner.size());
    return ISC_OK;
}

int ensure_bytes(void **p, size_t *have, size_t need)
{
    if (*have >= need && *p) return ISC_OK;
    if (*p) cudaFree(*p);
    *p = nullptr; *have = 0;
    CK(cudaMalloc(p, std::max<size_t>(need, 16)));
    *have = need;
    return ISC_OK;
}

void free_workspace(isc_model *m)
{
    for (DevBuf &b : m->bufs) {
        if (b.p) cudaFree(b.p);
        b = DevBuf();
    }
    m->ws_batch = 0;
}

int ensure_workspace(isc_model *m, int batch)
{
    if (batch <= m->ws_batch) return ISC_OK;
    free_workspace(m);
    for (size_t b = 0; b < m->bufs.size(); ++b) {
        const cudaError_t e = cudaMalloc(&m->bufs[b].p, m->buf_bytes[b] * (size_t)batch);
        if (e != cudaSuccess) {
            m->bufs[b].p = nullptr;
            free_workspace(m);
            CK(e);
        }
        m->bufs[b].bytes = m->buf_bytes[b] * (size_t)batch;
    }
    m->ws_batch = batch;
    return ISC_OK;
}

// Appends the table of bins at `bits` bits to the tables at `tab`, which begin with the cumulative one; false, and nothing
// appended, if more than one uniform in 2^11 lies in an open bin: the 128 of a warp share the way out, which then costs what the
// bins save (sixteen warps in all meet one).  The boundaries are counted per bin, from the middle of the range outwards, so that a
// vain try ends at once: where bins are too wide for the law, those in the middle are.  (Looking up both ends of every
// bin, in up to three full tries, took 37 us of a call with a new standard deviation of 1; this takes 14.)
bool noise_bins(std::vector<uint32_t> &tab, size_t n_cum, int bits)
{
    const uint32_t side = isc::noise_bins_side(bits), one = 1u << bits, from = 1u << isc::kNoiseBinsFrom, limit = 1u << 21;
    const size_t front = tab.size();
    const uint32_t n_bounds = (uint32_t)n_cum - 1;                       // level i + 1 begins at cum[i]
    const uint32_t middle = std::min((uint32_t)(std::upper_bound(tab.begin(), tab.begin() + n_cum, 0x7FFFFFFFu) - tab.begin()), n_bounds);
    // uniforms of bin b: all but the last bins are 2^e of them
    auto size_of = [&](uint32_t b) {
        const int e = isc::kNoiseBinsFrom + (int)(b >> bits) - bits;
        return e + bits < 31 ? 1u << e : b == side - 2 ? from : 0u;      // sums from 2^31 on: one bin up to 2^31 + 2^21, none beyond
    };
    // per bin: boundaries between two of its uniforms; between its first one (as counted from the end) and the bin before
    std::vector<uint16_t> counts(4 * (size_t)side, 0);
    uint64_t open = 0;
    for (uint32_t upper = 0; upper < 2; ++upper) {
        uint16_t *inside = counts.data() + 2 * (size_t)upper * side, *before = inside + side;
        const uint32_t n = upper ? n_bounds - middle : middle;
        for (uint32_t k = 0; k < n; ++k) {
            const uint32_t c = tab[upper ? middle + k : middle - 1 - k], first = upper ? 0u - c : c;       // the bound's larger distance from the end
            if (first > 0x7FFFFFFFu) continue;                           // between the two sides
            const uint32_t v = first + from;
            if (v < from + (from >> bits)) {                             // the outermost bin: the rest of the tail lies in it
                before[0] = upper ? 0 : (uint16_t)(std::upper_bound(tab.begin(), tab.begin() + n_cum, 0u) - tab.begin());
                inside[0] = (uint16_t)(n - k - before[0]);
                if (inside[0] > 1) open += size_of(0);
                break;
            }
            const int e = 31 - __builtin_clz(v) - bits;
            const uint32_t b = ((uint32_t)(e + bits - isc::kNoiseBinsFrom) << bits) + (v >> e) - one;
            if ((v & ((1u << e) - 1)) == 0) before[b] += 1;
            else if (++inside[b] == 2 && (open += size_of(b)) > limit) return false;
        }
    }
    tab.resize(front + 4 * (size_t)side);
    const uint32_t *cum = tab.data();
    const uint32_t T = n_bounds / 2;
    for (uint32_t upper = 0; upper < 2; ++upper) {
        const uint16_t *inside = counts.data() + 2 * (size_t)upper * side, *before = inside + side;
        uint32_t *entry = tab.data() + front + 2 * (size_t)upper * side;
        uint32_t at = upper ? n_bounds : 0;                              // the level from where the bins come from
        for (uint32_t b = 0; b < side; ++b, entry += 2) {
            const uint32_t low = upper ? at - before[b] - inside[b] : at + before[b];       // level of its smallest uniform
            at = upper ? low : low + inside[b];
            entry[0] = cum[low];
            entry[1] = low - T;
            if (inside[b] <= 1 && low != n_bounds) continue;
            if (inside[b] <= 1) open += size_of(b);                                         // the last level has no boundary above it
            entry[0] = 0;
            entry[1] = (uint32_t)isc::kNoiseOpen;
        }
        entry[-2] = 0;                                                                      // no uniform has the last bin
        entry[-1] = (uint32_t)isc::kNoiseOpen;
    }
    if (open > limit) tab.resize(front);
    return open <= limit;
}

// The noise law's table for `sigma` on the host, kept for the next call.
void host_noise_table(isc_model *m, double sigma)
{
    if (m->tab_sigma == sigma && m->tab_kind == (int)m->opt_noise) return;
    std::vector<uint32_t> &cum = m->h_tab;
    m->tab_sigma = -1.0;
    cum.reserve((size_t)(2 * noise_halfwidth(sigma) + 1) + (isc::kNoiseGuide + 1) + 3 + 4 * (size_t)isc::noise_bins_side(8));
    if (m->opt_noise) noise_table_rounded(sigma, cum); else noise_table(sigma, cum);
    // the guide table and the bins follow the cumulative one in the same allocation
    const size_t n_cum = cum.size();
    uint32_t i = 0;
    for (int j = 0; j <= isc::kNoiseGuide; ++j) {
        const uint64_t u = (uint64_t)j << (32 - isc::kNoiseGuideBits);
        while (i + 1 < n_cum && u >= cum[i]) ++i;        // min{ i : u < cum[i] }, the last entry matching always
        cum.push_back(i);
    }
    m->tab_T = (int)(n_cum - 1) / 2;
    // bisection steps that close the widest guide interval
    uint32_t span = 0;
    for (int j = 0; j < isc::kNoiseGuide; ++j) span = std::max(span, cum[n_cum + j + 1] - cum[n_cum + j]);
    m->tab_steps = 0;
    while ((1u << m->tab_steps) < span + 1) ++m->tab_steps;
    m->tab_front = (cum.size() + 3) & ~(size_t)3;
    cum.resize(m->tab_front, 0);
    m->tab_bin_bits = 0;
    for (int bits = 6; bits <= 8 && !m->tab_bin_bits; ++bits)
        if (noise_bins(cum, n_cum, bits)) m->tab_bin_bits = bits;
    m->tab_sigma = sigma;
    m->tab_kind = (int)m->opt_noise;
}

int ensure_noise_table(isc_model *m, double sigma, cudaStream_t st)
{
    host_noise_table(m, sigma);
    if (m->d_cum && m->cum_sigma == sigma && m->cum_kind == (int)m->opt_noise) return ISC_OK;
    size_t have = m->d_cum_n * sizeof(uint32_t);
    void *p = m->d_cum;
    int rc = ensure_bytes(&p, &have, m->h_tab.size() * sizeof(uint32_t));
    m->d_cum = (uint32_t *)p; m->d_cum_n = have / sizeof(uint32_t);
    if (rc) return rc;
    CK(cudaMemcpyAsync(m->d_cum, m->h_tab.data(), m->h_tab.size() * sizeof(uint32_t), cudaMemcpyHostToDevice, st));
    CK(cudaStreamSynchronize(st));                       // the host table may change
    m->cum_sigma = sigma;
    m->cum_kind = (int)m->opt_noise;
    return ISC_OK;
}

int check_stream_args(uint64_t image_id, int32_t phase, int64_t first, int64_t n, double sigma)
{
    if (!(sigma > 0.0) || !std::isfinite(sigma) || sigma > 64.0) return ISC_ERR_ARG;
    if (phase < 0 || phase > 255) return ISC_ERR_ARG;
    if (image_id >= (1ull << 48)) return ISC_ERR_ARG;
    if (first < 0 || n < 0 || first + n > (1ll << 40)) return ISC_ERR_ARG;
    return ISC_OK;
}

int check_certify_args(uint64_t last_image_id, int64_t N0, int64_t N, double sigma, double alpha)
{
    if (N0 < 1 || N < 1 || !(alpha > 0.0 && alpha < 1.0)) return ISC_ERR_ARG;
    if (N0 > (1ll << 31) - 1 || N > (1ll << 31) - 1) return ISC_ERR_ARG;
    return check_stream_args(last_image_id, 0, 0, std::max(N0, N), sigma);
}

NoiseStream make_stream(const isc_model *m, uint64_t seed, uint64_t image_id, int32_t phase, int64_t first)
{
    NoiseStream ns;
    ns.key0 = (uint32_t)(seed & 0xFFFFFFFFu);
    ns.key1 = (uint32_t)(seed >> 32);
    ns.ctr2 = (uint32_t)(image_id & 0xFFFFFFFFu);
    ns.ctr3_fixed = (uint32_t)phase | (uint32_t)(((image_id >> 32) & 0xFFFFu) << 16);
    ns.first_sample = first;
    ns.cum = m->d_cum;
    ns.T = m->tab_T;
    ns.guide = m->d_cum ? m->d_cum + (2 * m->tab_T + 1) : nullptr;
    ns.guide_steps = m->tab_steps;
    ns.bins = m->d_cum && m->tab_bin_bits ? reinterpret_cast<const uint2 *>(m->d_cum + m->tab_front) : nullptr;
    ns.bin_bits = m->tab_bin_bits;
    return ns;
}

int choose_engine(isc_model *m)
{
    if (m->opt_engine == 1) return 1;
    if (m->opt_engine == 2) return m->has_tc ? 2 : ISC_ERR_UNSUPPORTED;
    if (m->opt_engine == 3) return m->line ? 3 : ISC_ERR_UNSUPPORTED;
    if (m->line) return 3;
    if (m->has_tc) return 2;
    return 1;
}

std::vector<int8_t *> own_buffers(const isc_model *m)
{
    std::vector<int8_t *> b;
    for (const DevBuf &d : m->bufs) b.push_back((int8_t *)d.p);
    return b;
}

int ready_tensor_cores(isc_model *m)
{
    int device = -1;
    CK(cudaGetDevice(&device));
    if (device != m->tc.ordinal) CK(tc_prepare(&m->tc, device));
    return ISC_OK;
}

// Layer-by-layer forward of `batch` samples in the activation buffers `bufs`; leaves the logits in the last tensor's.
// run: what the samples are (`ns`: only the seed and the tables).  `chained`: the stream's last operation is a kernel of such a forward too (see launch_chained).
int generic_forward(isc_model *m, int8_t *const *bufs, const uint8_t *d_x, const NoiseStream &ns, const SampleRun &run, int batch, cudaStream_t st, int32_t *d_err,
                    int stop_after_layer = -1, bool tensor_cores = false, bool chained = false)
{
    const int n = (int)m->glayers.size();
    if (tensor_cores) {
        int rc = ready_tensor_cores(m);
        if (rc) return rc;
    }
    const bool follows = tensor_cores && m->tc.chained;
    for (int i = 0; i < n; ++i) {
        const GLayer &G = m->glayers[(size_t)i];
        const isc_layer &L = m->layers[(size_t)i].d;
        int8_t *out = bufs[m->tensor_buf[(size_t)i + 1]];
        const int8_t *in = i == 0 ? nullptr : bufs[m->tensor_buf[(size_t)L.in_tensor]];
        const int8_t *res = L.res_tensor >= 0 ? bufs[m->tensor_buf[(size_t)L.res_tensor]] : nullptr;
        cudaError_t e;
        if (i == 0 && tensor_cores && m->wpacks[0])
            e = launch_stem_conv(m->tc, G, m->wpacks[0], m->tc_cst[0], m->tc_fast[0] != 0, d_x, m->in_c, ns, run, batch, out, d_err, st, false, chained);
        else if (i == 0) e = launch_first_conv(G, d_x, m->in_c, ns, run, batch, out, st);
        else if (tensor_cores && m->hpacks[(size_t)i] && halo_offsets_fit(G, batch))
            e = launch_halo_conv(m->tc, G, m->hpacks[(size_t)i], m->tc_cst[(size_t)i], m->tc_fast[(size_t)i] != 0, m->tc_resk[(size_t)i], batch, in, res, out, d_err, st);
        else if (tensor_cores && m->wpacks[(size_t)i] && conv_offsets_fit(G, batch)) e = launch_igemm_conv(m->tc, G, m->wpacks[(size_t)i], m->tc_cst[(size_t)i], m->tc_fast[(size_t)i] != 0, m->tc_resk[(size_t)i], batch, in, res, out, d_err, st, false, m->opt_tensor_copy != 0);
        else if (L.op == ISC_CONV2D || L.op == ISC_FC) e = launch_conv(G, batch, in, res, out, st);
        else if (L.op == ISC_GAVGPOOL) e = launch_gavgpool(G, batch, in, out, st, follows);
        else e = launch_maxpool(G, batch, in, out, st, follows);
        m->launches += 1;
        if (e != cudaSuccess) {
            if (getenv("ISC_DEBUG_CUDA")) fprintf(stderr, "isc: layer %d launch: %s\n", i, cudaGetErrorString(e));
            return ISC_ERR_CUDA;
        }
        if (i == stop_after_layer) break;
    }
    return ISC_OK;
}

size_t generic_bytes_per_sample(const isc_model *m)
{
    size_t s = 0;
    for (size_t b : m->buf_bytes) s += b;
    return s;
}

// The Monte-Carlo loop on the layer-by-layer kernels: `total` samples of `run`, in equal batches of at most `cap`, in the
// activation buffers `bufs`; adds votes into d_counts (device).
int forward_counts(isc_model *m, int8_t *const *bufs, int64_t cap, bool tensor_cores, const uint8_t *d_x, const NoiseStream &ns, SampleRun run, int64_t total,
                   cudaStream_t st, int32_t *d_counts, int8_t *d_logits, int32_t *d_err)
{
    const int last = (int)m->glayers.size();
    const int64_t batches = (total + cap - 1) / cap, size = batches ? (total + batches - 1) / batches : 0, begin = (int64_t)run.first;
    for (int64_t done = 0; done < total; done += size) {
        const int b = (int)std::min<int64_t>(size, total - done);
        run.first = (uint64_t)(begin + done);
        int rc = generic_forward(m, bufs, d_x, ns, run, b, st, d_err, -1, tensor_cores, done > 0);
        if (rc) return rc;
        cudaError_t e = launch_votes(bufs[m->tensor_buf[(size_t)last]], m->shapes[(size_t)last].cp, m->n_classes, run, b, d_counts,
                                     d_logits ? d_logits + (size_t)done * m->n_classes : nullptr, st, tensor_cores && m->tc.chained);
        m->launches += 1;
        if (e != cudaSuccess) return ISC_ERR_CUDA;
    }
    return ISC_OK;
}

// Samples a batch may have: the tensor-core kernels' offsets are 32-bit.
int64_t tensor_core_cap(const isc_model *m)
{
    int64_t cap = 32768;
    for (size_t b : m->buf_bytes) cap = std::min<int64_t>(cap, std::max<int64_t>(1, (int64_t)(((1ull << 31) - 1) / std::max<size_t>(b, 1))));
    return cap;
}

// The samples of one phase of one image.
SampleRun one_phase(uint64_t image_id, int32_t phase, int64_t first, int64_t n)
{
    return SampleRun{image_id, 0, (uint64_t)std::max<int64_t>(n, 1), 0, (uint64_t)first, 0, (uint32_t)phase};
}

// Samples of a batch in the handle's own buffers.
int64_t layerwise_cap(const isc_model *m)
{
    int64_t cap = m->opt_batch > 0 ? m->opt_batch : 8192;
    const size_t per = std::max<size_t>(generic_bytes_per_sample(m), 1);
    cap = std::min<int64_t>(cap, std::max<int64_t>(1, (int64_t)((3ull << 30) / per)));
    return std::min<int64_t>(std::min(cap, m->ws_limit), m->last_engine == 2 ? tensor_core_cap(m) : 32768);
}

// forward_counts in the handle's own buffers.  Where the device's memory does not hold a batch, half of it and so on; the
// handle then keeps to what fitted, so that later calls do not try in vain.
int layerwise_counts(isc_model *m, const uint8_t *d_x, uint64_t seed, const SampleRun &run, int64_t total, cudaStream_t st, int32_t *d_counts, int8_t *d_logits, int32_t *d_err)
{
    int64_t cap = std::min<int64_t>(layerwise_cap(m), std::max<int64_t>(total, 1));
    int rc;
    while ((rc = ensure_workspace(m, (int)cap)) == ISC_ERR_NOMEM && cap > 1) m->ws_limit = cap = (cap + 1) / 2;
    if (rc) return rc;
    return forward_counts(m, own_buffers(m).data(), cap, m->last_engine == 2, d_x, make_stream(m, seed, 0, 0, 0), run, total, st, d_counts, d_logits, d_err);
}

constexpr size_t kCountsOff = 16;                        // of the counts in the call buffer: the error word comes first
constexpr size_t kStagedBytes = 4u << 20;                // larger uploads and downloads do not go through the pinned buffer

int ensure_pinned(isc_model *m, size_t need)
{
    if (m->h_io_bytes >= need) return ISC_OK;
    if (m->h_io) cudaFreeHost(m->h_io);
    m->h_io = nullptr; m->h_io_bytes = 0;
    need = (need + 4095) & ~(size_t)4095;
    CK(cudaHostAlloc((void **)&m->h_io, need, cudaHostAllocDefault));
    m->h_io_bytes = need;
    return ISC_OK;
}

// The start of a call: error word and `n_counts` counts cleared, the images on the device.  The kernels read images as
// 32-bit words where an image row is whole words; device images that are not aligned for that are copied like host images.
int begin_call(isc_model *m, const uint8_t *x, size_t x_bytes, bool x_on_device, size_t n_counts, cudaStream_t st, const uint8_t **d_x)
{
    const size_t head = kCountsOff + n_counts * sizeof(int32_t), x_off = (head + 15) & ~(size_t)15;
    const bool in_place = x_on_device && (uintptr_t)x % 4 == 0;
    void *p = m->d_io;
    int rc = ensure_bytes(&p, &m->d_io_bytes, x_off + (in_place ? 0 : x_bytes));
    m->d_io = (uint8_t *)p;
    if (rc) return rc;
    const bool staged = !x_on_device && x_off + x_bytes <= kStagedBytes;
    if ((rc = ensure_pinned(m, staged ? x_off + x_bytes : head))) return rc;
    if (staged) {
        memset(m->h_io, 0, x_off);
        memcpy(m->h_io + x_off, x, x_bytes);
        CK(cudaMemcpyAsync(m->d_io, m->h_io, x_off + x_bytes, cudaMemcpyHostToDevice, st));
    } else {
        CK(cudaMemsetAsync(m->d_io, 0, head, st));
        if (!in_place) CK(cudaMemcpyAsync(m->d_io + x_off, x, x_bytes, x_on_device ? cudaMemcpyDefault : cudaMemcpyHostToDevice, st));
    }
    *d_x = in_place ? x : m->d_io + x_off;
    return ISC_OK;
}
int32_t *call_err(isc_model *m) { return (int32_t *)m->d_io; }
int32_t *call_counts(isc_model *m) { return (int32_t *)(m->d_io + kCountsOff); }
const int32_t *host_counts(const isc_model *m) { return (const int32_t *)(m->h_io + kCountsOff); }

// The error word, then counts [first, first + n), back into the pinned buffer.
int fetch_counts(isc_model *m, size_t first, size_t n, cudaStream_t st)
{
    const size_t off = first ? kCountsOff + first * sizeof(int32_t) : 0, end = kCountsOff + (first + n) * sizeof(int32_t);
    CK(cudaMemcpyAsync(m->h_io + off, m->d_io + off, end - off, cudaMemcpyDeviceToHost, st));
    return ISC_OK;
}

// After the stream has been synchronised and the error word fetched: has a bounded wait of a tensor-core kernel expired?
int call_status(const isc_model *m)
{
    const int32_t e = *(const int32_t *)m->h_io;
    if (m->last_engine == 3) return isc::line_status(e);
    return e ? ISC_ERR_TIMEOUT : ISC_OK;
}

// Votes of `n_images` images, n_sel samples of phase 0 and n_est of phase 1 each; `decide(i, counts0, counts)` is called
// for image after image while the kernels of later ones are in flight.
template <typename Decide>
int count_images(isc_model *m, const uint8_t *x, bool x_on_device, int n_images, uint64_t seed, uint64_t image_id0, int64_t n_sel,
                 int64_t n_est, double sigma, cudaStream_t st, Decide decide)
{
    const int engine = choose_engine(m);
    if (engine < 0) return engine;
    m->last_engine = engine;
    const size_t C = (size_t)m->n_classes, d = (size_t)m->in_c * m->in_h * m->in_w;
    int rc;
    if ((rc = ensure_noise_table(m, sigma, st))) return rc;
    const uint8_t *d_x;
    if ((rc = begin_call(m, x, d * (size_t)n_images, x_on_device, 2 * C * (size_t)n_images, st, &d_x))) return rc;
    // Pieces of the batch: as many images as make some sixty rounds of the resident engine's groups, so that a launch's
    // last, partly empty round costs little, or one batch of the layer-by-layer kernels, whose launches both phases and
    // several images share (a wide ResNet's 100 + 5,000 samples took three chains of launches, of 100, 4,096 and 904; in
    // one it is 2,794 -> 2,505 us).  The host's bounds still run under the next piece's kernels.
    const int64_t at_once = engine == 3 ? 64 * isc::line_wave_samples(m->line) : layerwise_cap(m);
    const int piece = (int)std::max<int64_t>(1, std::min<int64_t>(n_images, at_once / (n_sel + n_est)));
    const int n_pieces = (n_images + piece - 1) / piece;
    while ((int)m->events.size() < n_pieces - 1) {
        cudaEvent_t ev;
        CK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        m->events.push_back(ev);
    }
    for (int k = 0; k < n_pieces && rc == ISC_OK; ++k) {
        const int i0 = k * piece, n = std::min(piece, n_images - i0);
        int32_t *c = call_counts(m) + (size_t)i0 * 2 * C;
        if (engine == 3) {
            const isc::LineWork w{d_x + (size_t)i0 * d, n, image_id0 + (uint64_t)i0, n_sel, n_est, 0, c, nullptr};
            rc = isc::line_run(m->line, w, make_stream(m, seed, 0, 1, 0), (int)m->opt_batch, call_err(m), st, &m->launches);
        } else {
            const SampleRun run{image_id0 + (uint64_t)i0, (uint64_t)n_sel, (uint64_t)(n_sel + n_est), 0, 0, 0, 1};
            rc = layerwise_counts(m, d_x + (size_t)i0 * d, seed, run, (int64_t)n * (n_sel + n_est), st, c, nullptr, call_err(m));
        }
        if (rc == ISC_OK) rc = fetch_counts(m, (size_t)i0 * 2 * C, (size_t)n * 2 * C, st);
        if (rc == ISC_OK && k + 1 < n_pieces && cudaEventRecord(m->events[(size_t)k], st) != cudaSuccess) { cudaGetLastError(); rc = ISC_ERR_CUDA; }
    }
    if (rc == ISC_OK && n_pieces > 1 && cudaMemcpyAsync(m->h_io, m->d_io, kCountsOff, cudaMemcpyDeviceToHost, st) != cudaSuccess) { cudaGetLastError(); rc = ISC_ERR_CUDA; }
    if (rc) { cudaStreamSynchronize(st); return rc; }
    for (int k = 0; k < n_pieces; ++k) {
        CK(k + 1 < n_pieces ? cudaEventSynchronize(m->events[(size_t)k]) : cudaStreamSynchronize(st));
        for (int i = k * piece; i < std::min(n_images, (k + 1) * piece); ++i) {
            const int32_t *c0 = host_counts(m) + (size_t)i * 2 * C;
            decide(i, c0, c0 + C);
        }
    }
    return call_status(m);
}

// One launch of the tensor-core kernel that takes layer `li`, on one sample's work space, with the weights held back: the
// kernel's own waits run out and its CTAs leave through the abort path; the error word must be up afterwards.
int stalled_launch(isc_model *m, size_t li, cudaStream_t st, int32_t *err, int32_t *ns)
{
    if (!m->wpacks[li] && !m->hpacks[li]) return ISC_ERR_UNSUPPORTED;
    const GLayer &G = m->glayers[li];
    const isc_layer &L = m->layers[li].d;
    const uint8_t *d_x = nullptr;
    int rc = ensure_workspace(m, 1);
    if (rc == ISC_OK) rc = ready_tensor_cores(m);
    if (rc == ISC_OK && li == 0) {                           // the stem draws its noise first: on an empty image
        const std::vector<uint8_t> x((size_t)m->in_c * m->in_h * m->in_w, 0);
        rc = ensure_noise_table(m, 0.25, st);
        if (rc == ISC_OK) rc = begin_call(m, x.data(), x.size(), false, (size_t)m->n_classes, st, &d_x);
        if (rc == ISC_OK) CK(cudaStreamSynchronize(st));
    }
    if (rc) return rc;
    if (!m->d_tc_err) {
        const int32_t *p = nullptr;
        if ((rc = upload(m, std::vector<int32_t>(1, 0), &p))) return rc;
        m->d_tc_err = const_cast<int32_t *>(p);
    }
    int8_t *out = (int8_t *)m->bufs[(size_t)m->tensor_buf[li + 1]].p;
    const int8_t *in = li ? (const int8_t *)m->bufs[(size_t)m->tensor_buf[(size_t)L.in_tensor]].p : nullptr;
    const int8_t *res = L.res_tensor >= 0 ? (const int8_t *)m->bufs[(size_t)m->tensor_buf[(size_t)L.res_tensor]].p : nullptr;
    const bool fast = m->tc_fast[li] != 0;
    const auto t0 = std::chrono::steady_clock::now();
    cudaError_t e;
    if (li == 0) e = launch_stem_conv(m->tc, G, m->wpacks[0], m->tc_cst[0], fast, d_x, m->in_c, make_stream(m, 1, 0, 1, 0), SampleRun{0, 0, 1, 0, 0, 0, 1}, 1, out, m->d_tc_err, st, true);
    else if (m->hpacks[li]) e = launch_halo_conv(m->tc, G, m->hpacks[li], m->tc_cst[li], fast, m->tc_resk[li], 1, in, res, out, m->d_tc_err, st, true);
    else e = launch_igemm_conv(m->tc, G, m->wpacks[li], m->tc_cst[li], fast, m->tc_resk[li], 1, in, res, out, m->d_tc_err, st, true);
    if (e != cudaSuccess) return ISC_ERR_CUDA;
    CK(cudaStreamSynchronize(st));
    const long long t = std::chrono::duration_cast<std::chrono::nanoseconds>(std::chrono::steady_clock::now() - t0).count();
    CK(cudaMemcpy(err, m->d_tc_err, sizeof(*err), cudaMemcpyDeviceToHost));
    CK(cudaMemset(m->d_tc_err, 0, sizeof(*err)));
    *ns = (int32_t)std::min<long long>(t, 0x7FFFFFFF);
    return *err != 0 ? ISC_ERR_TIMEOUT : ISC_OK;
}

}  // namespace

// =============================================================================== C ABI

extern "C" {

const char *isc_strerror(int code)
{
    switch (code) {
    case ISC_OK: return "ok";
    case ISC_ERR_ARG: return "invalid argument";
    case ISC_ERR_SHAPE: return "layer list does not type-check";
    case ISC_ERR_UNSUPPORTED: return "not supported by the kernels";
    case ISC_ERR_NOMEM: return "out of memory";
    case ISC_ERR_CUDA: return "CUDA error";
    case ISC_ERR_TIMEOUT: return "device-side wait timed out";
    default: return "unknown error";
    }
}

int isc_load_qmodel(const isc_layer *layers, int n_layers, int in_c, int in_h, int in_w, int n_classes,
                    isc_model **out)
{
    if (!layers || !out || n_layers < 1 || n_layers > 4096) return ISC_ERR_ARG;
    if (in_c < 1 || in_h < 1 || in_w < 1 || n_classes < 1 || n_classes > 4096) return ISC_ERR_ARG;
    if ((int64_t)in_c * in_h * in_w > (1ll << 30)) return ISC_ERR_ARG;
    isc_model *m = new (std::nothrow) isc_model();
    if (!m) return ISC_ERR_NOMEM;
    m->in_c = in_c; m->in_h = in_h; m->in_w = in_w; m->n_classes = n_classes;
    int rc;
    try {
        rc = build_host_model(m, layers, n_layers);
        if (rc == ISC_OK) rc = build_generic_engine(m);
        if (rc == ISC_OK) {
            std::vector<isc::LayerIn> ml(m->layers.size());
            for (size_t i = 0; i < m->layers.size(); ++i) {
                const HostLayer &H = m->layers[i];
                ml[i].d = H.d;
                ml[i].w = H.w.data(); ml[i].bias = H.bias.data();
                ml[i].mult = H.mult.data(); ml[i].shift = H.shift.data();
            }
            rc = isc::line_build(ml.data(), (int)ml.size(), in_c, in_h, in_w, n_classes, &m->line);
        }
    } catch (const std::bad_alloc &) {
        rc = ISC_ERR_NOMEM;
    }
    if (rc != ISC_OK) {
        isc_free_qmodel(m);
        return rc;
    }
    *out = m;
    return ISC_OK;
}

int isc_plan_resident(const isc_layer *layers, int n_layers, int in_c, int in_h, int in_w, int n_classes,
                      int32_t *out_rule, int64_t *out_smem_bytes)
{
    if (!layers || n_layers < 1 || n_layers > 4096) return ISC_ERR_ARG;
    if (in_c < 1 || in_h < 1 || in_w < 1 || n_classes < 1 || n_classes > 4096) return ISC_ERR_ARG;
    if ((int64_t)in_c * in_h * in_w > (1ll << 30)) return ISC_ERR_ARG;
    try {
        isc_model m;
        m.in_c = in_c; m.in_h = in_h; m.in_w = in_w; m.n_classes = n_classes;
        int rc = build_host_model(&m, layers, n_layers);
        if (rc) return rc;
        std::vector<isc::LayerIn> ml(m.layers.size());
        for (size_t i = 0; i < m.layers.size(); ++i) {
            const HostLayer &H = m.layers[i];
            ml[i].d = H.d;
            ml[i].w = H.w.data(); ml[i].bias = H.bias.data();
            ml[i].mult = H.mult.data(); ml[i].shift = H.shift.data();
        }
        int rule = 0;
        uint32_t smem = 0;
        const int fits = isc::line_plan_probe(ml.data(), (int)ml.size(), in_c, in_h, in_w, n_classes, &rule, &smem);
        if (out_rule) *out_rule = rule;
        if (out_smem_bytes) *out_smem_bytes = smem;
        return fits;
    } catch (const std::bad_alloc &) {
        return ISC_ERR_NOMEM;
    }
}

void isc_free_qmodel(isc_model *m)
{
    if (!m) return;
    for (void *p : m->param_allocs) cudaFree(p);
    for (DevBuf &b : m->bufs) if (b.p) cudaFree(b.p);
    if (m->d_io) cudaFree(m->d_io);
    if (m->d_logits) cudaFree(m->d_logits);
    if (m->d_cum) cudaFree(m->d_cum);
    if (m->h_io) cudaFreeHost(m->h_io);
    for (cudaEvent_t ev : m->events) cudaEventDestroy(ev);
    isc::line_free(m->line);
    delete m;
}

int isc_sample_counts(isc_model *m, const uint8_t *x_u8, uint64_t seed, uint64_t image_id, int32_t phase,
                      int64_t first_sample, int64_t n_samples, double sigma, void *cuda_stream,
                      int32_t *out_counts, int8_t *out_logits)
{
    if (!m || !x_u8 || !out_counts) return ISC_ERR_ARG;
    int rc = check_stream_args(image_id, phase, first_sample, n_samples, sigma);
    if (rc) return rc;
    if (n_samples > (1ll << 31) - 1) return ISC_ERR_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int engine = choose_engine(m);
    if (engine < 0) return engine;
    m->last_engine = engine;
    const size_t C = (size_t)m->n_classes;
    const size_t logit_bytes = out_logits ? (size_t)n_samples * C : 0;
    const size_t logits_off = kCountsOff + C * sizeof(int32_t);          // in the pinned buffer
    const bool staged = logits_off + logit_bytes <= kStagedBytes;
    if ((rc = ensure_noise_table(m, sigma, st))) return rc;
    if ((rc = ensure_pinned(m, logits_off + (staged ? logit_bytes : 0)))) return rc;
    if (out_logits) {
        void *p = m->d_logits; size_t have = m->d_logits_bytes;
        rc = ensure_bytes(&p, &have, std::max<size_t>(logit_bytes, C));
        m->d_logits = (int8_t *)p; m->d_logits_bytes = have;
        if (rc) return rc;
    }
    const uint8_t *d_x;
    if ((rc = begin_call(m, x_u8, (size_t)m->in_c * m->in_h * m->in_w, false, C, st, &d_x))) return rc;
    int8_t *d_logits = out_logits ? m->d_logits : nullptr;
    if (engine == 3) {
        const isc::LineWork w{d_x, 1, image_id, 0, n_samples, 0, call_counts(m), d_logits};
        rc = isc::line_run(m->line, w, make_stream(m, seed, 0, phase, first_sample), (int)m->opt_batch, call_err(m), st, &m->launches);
    } else {
        rc = layerwise_counts(m, d_x, seed, one_phase(image_id, phase, first_sample, n_samples), n_samples, st, call_counts(m), d_logits, call_err(m));
    }
    if (rc) {
        cudaStreamSynchronize(st);
        return rc;
    }
    if ((rc = fetch_counts(m, 0, C, st))) return rc;
    std::vector<int8_t> hl;
    const int8_t *h_logits = (const int8_t *)m->h_io + logits_off;
    if (logit_bytes) {
        if (!staged) {
            hl.resize(logit_bytes);
            h_logits = hl.data();
        }
        CK(cudaMemcpyAsync(const_cast<int8_t *>(h_logits), m->d_logits, logit_bytes, cudaMemcpyDeviceToHost, st));
    }
    CK(cudaStreamSynchronize(st));
    if ((rc = call_status(m))) return rc;
    memcpy(out_counts, host_counts(m), C * sizeof(int32_t));
    if (logit_bytes) memcpy(out_logits, h_logits, logit_bytes);
    return ISC_OK;
}

int isc_predict(isc_model *m, const uint8_t *x_u8, uint64_t seed, uint64_t image_id, int64_t N, double sigma,
                double alpha, void *cuda_stream, int32_t *out_class, int32_t *out_counts)
{
    if (!m || !x_u8 || !out_class) return ISC_ERR_ARG;
    if (N < 1 || !(alpha > 0.0 && alpha < 1.0)) return ISC_ERR_ARG;
    std::vector<int32_t> counts((size_t)m->n_classes);
    int rc = isc_sample_counts(m, x_u8, seed, image_id, 2, 0, N, sigma, cuda_stream, counts.data(), nullptr);
    if (rc) return rc;
    *out_class = decide_predict(counts.data(), m->n_classes, alpha);
    if (out_counts) memcpy(out_counts, counts.data(), counts.size() * sizeof(int32_t));
    return ISC_OK;
}

int isc_certify_batch(isc_model *m, const uint8_t *x_u8, int x_on_device, int n_images, uint64_t seed,
                      uint64_t image_id0, int64_t N0, int64_t N, double sigma, double alpha, void *cuda_stream,
                      int32_t *out_class, double *out_radius, int32_t *out_counts0, int32_t *out_counts)
{
    if (!m || !x_u8 || !out_class || !out_radius || n_images < 0) return ISC_ERR_ARG;
    int rc = check_certify_args(image_id0 + (uint64_t)std::max(n_images - 1, 0), N0, N, sigma, alpha);
    if (rc) return rc;
    if (n_images == 0) return ISC_OK;
    const size_t C = (size_t)m->n_classes;
    std::vector<int32_t> cls((size_t)n_images, -1);
    std::vector<double> rad((size_t)n_images, 0.0);
    rc = count_images(m, x_u8, x_on_device != 0, n_images, seed, image_id0, N0, N, sigma, (cudaStream_t)cuda_stream,
                      [&](int i, const int32_t *c0, const int32_t *c1) {
                          cls[(size_t)i] = decide_certify(c0, c1, m->n_classes, N, sigma, alpha, &rad[(size_t)i], nullptr);
                      });
    if (rc) return rc;
    for (int i = 0; i < n_images; ++i) {
        const int32_t *c0 = host_counts(m) + (size_t)i * 2 * C, *c1 = c0 + C;
        out_class[i] = cls[(size_t)i];
        out_radius[i] = rad[(size_t)i];
        if (out_counts0) memcpy(out_counts0 + (size_t)i * C, c0, C * sizeof(int32_t));
        if (out_counts) memcpy(out_counts + (size_t)i * C, c1, C * sizeof(int32_t));
    }
    return ISC_OK;
}

int isc_certify(isc_model *m, const uint8_t *x_u8, uint64_t seed, uint64_t image_id, int64_t N0, int64_t N,
                double sigma, double alpha, void *cuda_stream, int32_t *out_class, double *out_radius,
                int32_t *out_counts0, int32_t *out_counts)
{
    return isc_certify_batch(m, x_u8, 0, 1, seed, image_id, N0, N, sigma, alpha, cuda_stream, out_class,
                             out_radius, out_counts0, out_counts);
}

int isc_decide_certify(const int32_t *counts0, const int32_t *counts, int n_classes, int64_t N, double sigma,
                       double alpha, int32_t *out_class, double *out_radius, double *out_p_lower)
{
    if (!counts0 || !counts || !out_class || !out_radius || n_classes < 1 || N < 1) return ISC_ERR_ARG;
    if (!(alpha > 0.0 && alpha < 1.0) || !(sigma > 0.0)) return ISC_ERR_ARG;
    for (int c = 0; c < n_classes; ++c)
        if (counts0[c] < 0 || counts[c] < 0 || counts[c] > N) return ISC_ERR_ARG;
    double radius = 0.0, pl = 0.0;
    *out_class = decide_certify(counts0, counts, n_classes, N, sigma, alpha, &radius, &pl);
    *out_radius = radius;
    if (out_p_lower) *out_p_lower = pl;
    return ISC_OK;
}

int isc_decide_certify_integer(const int32_t *counts0, const int32_t *counts, int n_classes, int64_t N, double sigma,
                               double alpha, int two_sided, int32_t *out_class, int32_t *out_q, int64_t *out_q_squared)
{
    if (!counts0 || !counts || !out_class || !out_q || n_classes < 1 || N < 1) return ISC_ERR_ARG;
    if (!(alpha > 0.0 && alpha < 1.0) || !(sigma > 0.0) || !std::isfinite(sigma) || sigma > 64.0) return ISC_ERR_ARG;
    for (int c = 0; c < n_classes; ++c)
        if (counts0[c] < 0 || counts[c] < 0 || counts[c] > N) return ISC_ERR_ARG;
    int32_t q = 0;
    int64_t q2 = 0;
    *out_class = decide_certify_integer(counts0, counts, n_classes, N, sigma, alpha, two_sided != 0, &q, &q2, nullptr, 0);
    *out_q = q;
    if (out_q_squared) *out_q_squared = q2;
    return ISC_OK;
}

int isc_certify_integer(isc_model *m, const uint8_t *x_u8, uint64_t seed, uint64_t image_id, int64_t N0, int64_t N,
                        double sigma, double alpha, int two_sided, void *cuda_stream, int32_t *out_class,
                        int32_t *out_q, int64_t *out_q_squared, int32_t *out_counts0, int32_t *out_counts)
{
    if (!m || !x_u8 || !out_class || !out_q) return ISC_ERR_ARG;
    int rc = check_certify_args(image_id, N0, N, sigma, alpha);
    if (rc) return rc;
    const size_t C = (size_t)m->n_classes;
    int32_t cls = -1, q = 0;
    int64_t q2 = 0;
    rc = count_images(m, x_u8, false, 1, seed, image_id, N0, N, sigma, (cudaStream_t)cuda_stream,
                      [&](int, const int32_t *c0, const int32_t *c1) {
                          // the handle's table is Eq. 2's unless it draws from the rounded law
                          cls = decide_certify_integer(c0, c1, m->n_classes, N, sigma, alpha, two_sided != 0, &q, &q2,
                                                       m->tab_kind == 0 ? m->h_tab.data() : nullptr, 2 * m->tab_T + 1);
                      });
    if (rc) return rc;
    *out_class = cls;
    *out_q = q;
    if (out_q_squared) *out_q_squared = q2;
    if (out_counts0) memcpy(out_counts0, host_counts(m), C * sizeof(int32_t));
    if (out_counts) memcpy(out_counts, host_counts(m) + C, C * sizeof(int32_t));
    return ISC_OK;
}

int isc_decide_predict(const int32_t *counts, int n_classes, double alpha, int32_t *out_class)
{
    if (!counts || !out_class || n_classes < 1 || !(alpha > 0.0 && alpha < 1.0)) return ISC_ERR_ARG;
    for (int c = 0; c < n_classes; ++c)
        if (counts[c] < 0) return ISC_ERR_ARG;
    *out_class = decide_predict(counts, n_classes, alpha);
    return ISC_OK;
}

int isc_noise_table(double sigma, uint32_t *cum, int64_t capacity, int32_t *out_T)
{
    if (!out_T || !(sigma > 0.0) || !std::isfinite(sigma) || sigma > 64.0) return ISC_ERR_ARG;
    const int T = noise_halfwidth(sigma);
    if (cum) {
        if (capacity < 2 * (int64_t)T + 1) return ISC_ERR_ARG;
        std::vector<uint32_t> t;
        noise_table(sigma, t);
        memcpy(cum, t.data(), t.size() * sizeof(uint32_t));
    }
    *out_T = T;
    return ISC_OK;
}

int isc_noise_table_rounded(double sigma, uint32_t *cum, int64_t capacity, int32_t *out_T)
{
    if (!out_T || !(sigma > 0.0) || !std::isfinite(sigma) || sigma > 64.0) return ISC_ERR_ARG;
    const int T = noise_halfwidth(sigma);
    if (cum) {
        if (capacity < 2 * (int64_t)T + 1) return ISC_ERR_ARG;
        std::vector<uint32_t> t;
        noise_table_rounded(sigma, t);
        memcpy(cum, t.data(), t.size() * sizeof(uint32_t));
    }
    *out_T = T;
    return ISC_OK;
}

int isc_certified_metrics(const int32_t *classes, const double *radii, const int32_t *labels, int64_t n,
                          const double *r, int n_r, double *out_cp, double *out_ca)
{
    if (!out_cp || n < 0 || n_r < 0 || (n > 0 && (!classes || !radii || !labels)) || (n_r > 0 && (!r || !out_ca)))
        return ISC_ERR_ARG;
    int64_t certified = 0;
    for (int64_t i = 0; i < n; ++i) certified += classes[i] != -1;
    std::vector<double> ca((size_t)n_r, 0.0);
    for (int t = 0; t < n_r; ++t) {
        int64_t hit = 0;
        for (int64_t i = 0; i < n; ++i) hit += classes[i] != -1 && classes[i] == labels[i] && radii[i] >= r[t];
        ca[(size_t)t] = certified ? (double)hit / (double)certified : 0.0;
    }
    *out_cp = n ? (double)certified / (double)n : 0.0;
    for (int t = 0; t < n_r; ++t) out_ca[t] = ca[(size_t)t];
    return ISC_OK;
}

int isc_radius_integer(double sigma, uint32_t p_fx, int32_t *out_q, int64_t *out_q_squared)
{
    if (!out_q || !(sigma > 0.0) || !std::isfinite(sigma) || sigma > 64.0) return ISC_ERR_ARG;
    std::vector<uint32_t> t;
    noise_table(sigma, t);
    const int32_t T = (int32_t)(t.size() - 1) / 2;
    // the table is non-decreasing: first entry that reaches p_fx
    const int32_t q = (int32_t)(std::lower_bound(t.begin(), t.end(), p_fx) - t.begin());
    const int32_t level = q > 2 * T ? T : q - T;
    *out_q = level;
    if (out_q_squared) *out_q_squared = (int64_t)level * (int64_t)level;
    return ISC_OK;
}

int isc_debug_tensor(isc_model *m, const uint8_t *x_u8, uint64_t seed, uint64_t image_id, int32_t phase,
                     int64_t j, double sigma, int tensor, void *cuda_stream, int32_t *out, int64_t capacity)
{
    if (!m || !x_u8 || !out || tensor < 0 || tensor > (int)m->layers.size()) return ISC_ERR_ARG;
    int rc = check_stream_args(image_id, phase, j, 1, sigma);
    if (rc) return rc;
    const TShape &s = m->shapes[(size_t)tensor];
    const size_t n = (size_t)s.c * s.h * s.w;
    if (capacity < (int64_t)n) return ISC_ERR_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if ((rc = ensure_noise_table(m, sigma, st))) return rc;
    const uint8_t *d_x;
    if ((rc = begin_call(m, x_u8, (size_t)m->in_c * m->in_h * m->in_w, false, (size_t)m->n_classes, st, &d_x))) return rc;
    NoiseStream ns = make_stream(m, seed, image_id, phase, j);
    if (m->opt_engine == 3) {       // read the tensor back from the resident engine
        if (!m->line) return ISC_ERR_UNSUPPORTED;
        std::vector<int32_t> tmp(n);
        rc = isc::line_debug_tensor(m->line, d_x, ns, tensor, tmp.data(), call_counts(m), st, &m->launches);
        if (rc) return rc;
        memcpy(out, tmp.data(), n * sizeof(int32_t));
        return ISC_OK;
    }
    if (tensor == 0) {
        int32_t *d_out = nullptr;
        CK(cudaMalloc((void **)&d_out, n * sizeof(int32_t)));
        cudaError_t e = launch_noisy_input(d_x, m->in_c, m->in_h, m->in_w, ns, 1, d_out, st);
        m->launches += 1;
        if (e == cudaSuccess) e = cudaMemcpyAsync(out, d_out, n * sizeof(int32_t), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        cudaFree(d_out);
        return e == cudaSuccess ? ISC_OK : ISC_ERR_CUDA;
    }
    if ((rc = ensure_workspace(m, 1))) return rc;
    if ((rc = generic_forward(m, own_buffers(m).data(), d_x, ns, one_phase(image_id, phase, j, 1), 1, st, call_err(m), tensor - 1, m->opt_engine == 2 || (m->opt_engine == 0 && m->has_tc)))) return rc;
    std::vector<int8_t> h((size_t)s.h * s.w * s.cp);
    CK(cudaMemcpyAsync(h.data(), m->bufs[(size_t)m->tensor_buf[(size_t)tensor]].p, h.size(),
                       cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    for (int c = 0; c < s.c; ++c)
        for (int y = 0; y < s.h; ++y)
            for (int x = 0; x < s.w; ++x)
                out[((size_t)c * s.h + y) * s.w + x] = h[((size_t)y * s.w + x) * s.cp + c];
    return ISC_OK;
}

int isc_debug_residual_product(int32_t res_mult, int32_t res_shift, int32_t zp_res, int32_t *k, float *m, int32_t *c)
{
    if (!k || !m || !c) return ISC_ERR_ARG;
    int32_t cc = 0;
    const isc::ResidualForm f = isc::residual_form(res_mult, res_shift, zp_res, &cc);
    if (!f.exists()) return 0;
    *k = (int32_t)(f.k8 >> 8);
    memcpy(m, &f.m_bits, sizeof(*m));
    *c = cc;
    return 1;
}

int isc_debug_residual_form(int32_t res_mult, int32_t res_shift, int32_t zp_res, int32_t *k, int32_t *c)
{
    if (!k || !c) return ISC_ERR_ARG;
    const int n = 31 - res_shift;
    if ((n != 31 && n != 32) || res_mult <= 0) return 0;
    const uint64_t m2 = (uint64_t)(uint32_t)res_mult << (32 - n);
    if (m2 >= (1ull << 32)) return 0;
    const int64_t r2 = ((1ll << (n - 1)) - (128ll + zp_res) * (int64_t)res_mult) * (1ll << (32 - n));
    for (uint32_t off = 0; off < 4096; ++off) {
        int64_t first = 0;
        bool same = true;
        for (uint32_t u = 0; u < 256 && same; ++u) {
            const int64_t want = ((int64_t)(u * m2) + r2) >> 32;                 // arithmetic shift: floor
            const int64_t got = (int64_t)(((uint64_t)(256u * off + u) * m2) >> 32);
            if (u == 0) first = got - want;
            same = got - want == first;
        }
        if (!same) continue;
        *k = (int32_t)off;
        *c = (int32_t)first;
        return 1;
    }
    return 0;
}

int isc_debug_wait_timeout(isc_model *m, int64_t limit_ns, void *cuda_stream, int32_t *out4)
{
    if (!m || !out4) return ISC_ERR_ARG;
    if (!m->line && m->has_tc) {
        // the layer-by-layer tensor-core engine: its first implicit-GEMM layer
        size_t li = 1;
        while (li < m->glayers.size() && !m->wpacks[li]) ++li;
        if (li >= m->glayers.size()) return ISC_ERR_UNSUPPORTED;
        int32_t e = 0, ns = 0;
        const int rc = stalled_launch(m, li, (cudaStream_t)cuda_stream, &e, &ns);
        if (rc != ISC_OK && rc != ISC_ERR_TIMEOUT) return rc;
        out4[0] = 0; out4[1] = 0; out4[2] = e; out4[3] = ns;
        return rc;
    }
    if (!m->line) return ISC_ERR_UNSUPPORTED;
    int32_t tmp[4] = {0, 0, 0, 0};
    const int rc = isc::line_wait_probe(m->line, limit_ns, tmp, (cudaStream_t)cuda_stream);
    if (rc == ISC_ERR_ARG || rc == ISC_ERR_CUDA) return rc;
    memcpy(out4, tmp, sizeof(tmp));
    return rc;
}

int isc_debug_stalled_launch(isc_model *m, int layer, void *cuda_stream, int32_t *out2)
{
    if (!m || !out2 || layer < 0 || layer >= (int)m->layers.size()) return ISC_ERR_ARG;
    int32_t e = 0, ns = 0;
    const int rc = stalled_launch(m, (size_t)layer, (cudaStream_t)cuda_stream, &e, &ns);
    if (rc != ISC_OK && rc != ISC_ERR_TIMEOUT) return rc;
    out2[0] = e; out2[1] = ns;
    return rc;
}

}  // extern "C"

// ------------------------------------------------------------------ allocation-free variant
//
// Work space of isc_sample_counts_static: one fixed array in the library's device image.  Every
// GPU on which the library is loaded carries it from module load until the process exits.
#define ISC_STATIC_SCRATCH_BYTES ((32u << 20) + 4096u)
static __device__ __align__(256) unsigned char g_static_scratch[ISC_STATIC_SCRATCH_BYTES];

namespace {

constexpr size_t kStaticCountsBytes = 16u << 10;     // up to 4096 classes
constexpr size_t kStaticTableBytes = 64u << 10;      // up to 16384 table entries (sigma up to ~4.5)
constexpr size_t kStaticImageBytes = 1u << 20;       // up to 1 MiB of input image
constexpr int kMaxDevices = 64;
unsigned char *g_static_ptr[kMaxDevices];            // device address of the array, per device ordinal

// The symbol name is only a host-side handle; the kernels need the array's device address,
// which the runtime reports per device.  Done once for each device, with that device current.
int static_scratch_base(unsigned char **base)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ISC_ERR_CUDA;
    if (!g_static_ptr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return ISC_ERR_CUDA;
        }
        g_static_ptr[dev] = static_cast<unsigned char *>(p);
    }
    *base = g_static_ptr[dev];
    return ISC_OK;
}

}  // namespace

extern "C" int isc_sample_counts_static(isc_model *m, const uint8_t *x_u8, uint64_t seed, uint64_t image_id,
                                        int32_t phase, int64_t first_sample, int64_t n_samples, double sigma,
                                        void *cuda_stream, int32_t *out_counts)
{
    if (!m || !x_u8 || !out_counts) return ISC_ERR_ARG;
    int rc = check_stream_args(image_id, phase, first_sample, n_samples, sigma);
    if (rc) return rc;
    if (n_samples > (1ll << 31) - 1) return ISC_ERR_ARG;
    const size_t C = (size_t)m->n_classes;
    const size_t d = (size_t)m->in_c * m->in_h * m->in_w;
    const int T = noise_halfwidth(sigma);
    const size_t per_sample = generic_bytes_per_sample(m) + 256 * m->buf_bytes.size();
    const size_t fixed = kStaticCountsBytes + kStaticTableBytes + kStaticImageBytes;          // (and 4 KiB for alignment and the error word)
    // sizes beyond the fixed work space are refused, never silently truncated
    if (C * sizeof(int32_t) > kStaticCountsBytes) return ISC_ERR_UNSUPPORTED;
    if ((size_t)(2 * T + 1) * sizeof(uint32_t) > kStaticTableBytes) return ISC_ERR_UNSUPPORTED;
    if (d > kStaticImageBytes) return ISC_ERR_UNSUPPORTED;
    if (per_sample > ISC_STATIC_SCRATCH_BYTES - fixed - 4096) return ISC_ERR_UNSUPPORTED;
    const int engine = choose_engine(m);
    if (engine < 0) return engine;

    unsigned char *base = nullptr;
    if ((rc = static_scratch_base(&base))) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // What goes up, as one copy: error word, vote counts (both zero: the array keeps whatever the previous call left),
    // noise table (the guide too where it fits, and for the engines that read them the bins), image.
    host_noise_table(m, sigma);
    const size_t n_cum = (size_t)(2 * T + 1);
    auto fits = [](size_t n) { return n * sizeof(uint32_t) <= kStaticTableBytes; };
    const size_t n_tab = engine >= 2 && fits(m->h_tab.size()) ? m->h_tab.size() : fits(m->tab_front) ? m->tab_front : n_cum;
    auto up16 = [](size_t v) { return (v + 15) & ~(size_t)15; };
    const size_t counts_off = 16, tab_off = counts_off + up16(C * sizeof(int32_t)), x_off = tab_off + up16(n_tab * sizeof(uint32_t));
    if (x_off + d > fixed + 4096) return ISC_ERR_UNSUPPORTED;
    std::vector<unsigned char> head(x_off + d, 0);
    memcpy(&head[tab_off], m->h_tab.data(), n_tab * sizeof(uint32_t));
    memcpy(&head[x_off], x_u8, d);
    CK(cudaMemcpyAsync(base, head.data(), head.size(), cudaMemcpyHostToDevice, st));
    int32_t *d_err = reinterpret_cast<int32_t *>(base), *d_counts = reinterpret_cast<int32_t *>(base + counts_off);
    const uint8_t *d_x = base + x_off;
    NoiseStream ns = make_stream(m, seed, image_id, phase, first_sample);
    ns.cum = reinterpret_cast<const uint32_t *>(base + tab_off);
    ns.T = T;
    ns.guide = n_tab > n_cum ? ns.cum + n_cum : nullptr;
    ns.guide_steps = n_tab > n_cum ? m->tab_steps : 0;
    ns.bins = n_tab > m->tab_front ? reinterpret_cast<const uint2 *>(ns.cum + m->tab_front) : nullptr;
    // (ResNet-20, 2,000 samples: 4.1 ms with the plain kernels, 0.53 ms on the resident engine.)
    // The resident engine needs no work space but this; the layer-by-layer kernels take their activation buffers from the
    // rest of the array, as many samples at a time as fit.
    if (engine == 3) {
        // (its parameters carry the image's number on their own)
        ns.ctr3_fixed = (uint32_t)phase;
        const isc::LineWork w{d_x, 1, image_id, 0, n_samples, 0, d_counts, nullptr};
        rc = isc::line_run(m->line, w, ns, 0, d_err, st, &m->launches);
    } else {
        const bool tensor_cores = engine == 2;
        const int64_t cap = std::min<int64_t>(tensor_cores ? tensor_core_cap(m) : 32768, (int64_t)((ISC_STATIC_SCRATCH_BYTES - fixed - 4096) / per_sample));
        std::vector<int8_t *> buf(m->buf_bytes.size());
        size_t off = fixed + 4096;
        for (size_t b = 0; b < buf.size(); ++b) {                    // 256-byte aligned
            buf[b] = reinterpret_cast<int8_t *>(base + off);
            off += (m->buf_bytes[b] * (size_t)cap + 255) & ~(size_t)255;
        }
        rc = forward_counts(m, buf.data(), cap, tensor_cores, d_x, ns, one_phase(image_id, phase, first_sample, n_samples), n_samples, st, d_counts, nullptr, d_err);
    }
    m->last_engine = 1;                 // "engine" has always read 1 after this entry point; "static_engine" tells which one ran
    m->last_static_engine = engine;
    if (rc) { cudaStreamSynchronize(st); return rc; }
    std::vector<int32_t> h(counts_off / sizeof(int32_t) + C);
    CK(cudaMemcpyAsync(h.data(), base, h.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (h[0]) return ISC_ERR_TIMEOUT;
    memcpy(out_counts, h.data() + counts_off / sizeof(int32_t), C * sizeof(int32_t));
    return ISC_OK;
}

extern "C" {

int isc_set_option(isc_model *m, const char *name, int64_t value)
{
    if (!m || !name) return ISC_ERR_ARG;
    if (!strcmp(name, "batch")) {
        if (value < 0 || value > (1 << 20)) return ISC_ERR_ARG;
        m->opt_batch = value;
        m->ws_limit = INT64_MAX;
        return ISC_OK;
    }
    if (!strcmp(name, "noise")) {
        if (value != 0 && value != 1) return ISC_ERR_ARG;
        m->opt_noise = value;
        return ISC_OK;
    }
    if (!strcmp(name, "tensor_copy")) {
        if (value != 0 && value != 1) return ISC_ERR_ARG;
        m->opt_tensor_copy = value;
        return ISC_OK;
    }
    if (!strcmp(name, "engine")) {
        if (value < 0 || value > 3) return ISC_ERR_ARG;
        m->opt_engine = value;
        return ISC_OK;
    }
    return ISC_ERR_ARG;
}

int isc_get_info(isc_model *m, const char *name, int64_t *out)
{
    if (!m || !name || !out) return ISC_ERR_ARG;
    if (!strcmp(name, "engine")) *out = m->last_engine;
    else if (!strcmp(name, "static_engine")) *out = m->last_static_engine;
    else if (!strcmp(name, "gpu_launches")) *out = m->launches;
    else if (!strcmp(name, "macs_per_sample")) *out = m->macs;
    else if (!strcmp(name, "has_line_engine")) *out = m->line ? 1 : 0;
    else if (!strcmp(name, "has_tensor_core_layers")) *out = m->has_tc ? 1 : 0;
    else if (!strncmp(name, "cycles_", 7)) {
        static const char *const which[4] = {"cycles_fill", "cycles_noise", "cycles_conv", "cycles_tail"};
        if (!m->line) return ISC_ERR_UNSUPPORTED;
        unsigned long long c[4];
        int rc = isc::line_phase_cycles(m->line, c);
        if (rc) return rc;
        for (int k = 0; k < 4; ++k)
            if (!strcmp(name, which[k])) { *out = (int64_t)c[k]; return ISC_OK; }
        return ISC_ERR_ARG;
    }
    else return ISC_ERR_ARG;
    return ISC_OK;
}

}  // extern "C"
