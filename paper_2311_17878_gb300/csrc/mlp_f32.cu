// Single-precision networks on the tcgen05 tensor cores: every operand as two FP16 parts.
//
// An FP32 operand x is carried as hi = fp16(32 x) and lo = fp16(2048 (32 x - hi)): 22
// significant bits over |x| from 2e-6 to 2047, and an absolute floor of 5e-13 below that (lo is
// stored scaled, so it stays normal while hi is).  A product sum takes three products per K step,
// hi hi' into a main accumulator and lo hi' + hi lo' into a correction accumulator that is
// scaled back by 2^-11 when it is read (lo lo' is below 2^-22 of the product).  Main and correction
// columns adjoin in TMEM and hi' and lo' rows in shared memory, so hi hi' and hi lo' are one MMA of
// twice the outputs: the hi operand is read once for both (20 instead of 24 KB of shared memory per K
// step; at 128 bytes a cycle the three MMAs alone took what the tensor cores need for them).  Everything
// between the products is FP32.
//
// tcgen05 truncates when it adds into its FP32 accumulator, so the main sum comes out too small
// by half a unit in the last place per MMA on average: measured against FP64 over random
// operands of either sign, 2.0e-8 + 1.67e-8 n of the sum after n MMAs with weights of 22 bits and
// 6 % less with weights of 8 (BF16 values), the same for positive and for signed rows.  The
// epilogue adds the mean of the two back (kBias0 + n kBias1).  What remains at K = 256 is
// 2.0e-7 (2-norm), an FP32 FMA chain has 2.9e-7; without the share 3.5e-7 and, worse, of one
// sign in every layer; with the three products in one accumulator 9.8e-7.  Through the fitted
// room networks: |grad f| 1.6e-7 off (FP32 FMA chains 3.0e-7; without the share 8.9e-7).
//
// Tile: 32 samples = 128 operand rows; TMEM lane quarter q holds samples 8q..8q+7 in four groups
// of 8 lanes (value, d/dx, d/dy, d/dz rows: forward-mode gradient).  Two parts of 128 x 256
// operands take 128 KB of shared memory.  A layer runs in phases of at most 128 outputs, each
// into one of two buffers of TMEM (main and correction, up to 128 columns each), so the epilogue of a
// phase runs beside the MMAs of the next.  A layer's operand can be replaced only after its last
// MMA: the first phase's activations wait in registers (as packed parts), are stored when the
// second phase is through, and the next layer starts on those 128 columns while the second
// phase's epilogue fills the others.  The narrow outputs, net_0 (with its gradient) and the
// three colours, are FP32 dot products that the epilogue of the layer before accumulates: no MMA
// phase of 16 columns with its hand-offs, and no truncation where |grad f| is near 1 everywhere
// and the mantissa would make the truncated share differ from its mean for every sample alike.  The weights stream from L2 in items of 64 K columns x
// 128 outputs (hi and lo, 32 KB) through a ring of two stages; three producer warps copy the
// items' parts in turn, because one thread's bulk copies do not overlap.
//
// The colour network has value rows only, a quarter of a tile's: so its layers run once for up to
// kUnit tiles, on all 128 rows.  Each tile's colour input (the SDF features, and x~, the
// direction encoding and the unit normal) is parked in global memory (L2) in operand layout, tile j
// in row group j of every lane quarter; bulk copies bring the features back as the operand, and
// the other columns through the weight ring as an item of their own before their weights.  (One
// tile at a time the colour layers were 38 of a tile's 96 items.)  61 915 samples of the room
// networks: SIMT kernel 13.8 ms, this one with the colour layers per tile 1.20 ms, per unit 1.10 ms,
// with the epilogue's groups two at a time 1.03 ms, one MMA for hi hi' and hi lo' 1.00 ms, and an
// item's MMAs as straight code 0.95 ms.  Of a tile's 145 k cycles the epilogue works for 86 k and
// the MMAs take 53 k at the tensor cores' rate; a layer's two phases overlap them in part.
//
// VALUE: the samplers' coarse pass (SDF value only): 128 samples per tile, one row each, no
// gradient and no colour network.
//
// Range: an operand beyond 2000, a non-finite value or a gradient below 1e-4 marks its sample
// (pad = 1 in its record; in the coarse pass a NaN of a fixed payload as its value) and a launch of
// the SIMT kernel evaluates the marked samples again: the split has no exponent range to spare there.
// So is, towards the floor, a sample with a hidden layer whose tangents (colours: activations) all lie
// below 1.9e-6, where the scaled high part is subnormal and the two have fewer than 22 bits; a layer
// whose weights do marks every sample.  Nothing is marked with networks of ordinary weights (the largest
// tangent of a hidden layer of the fitted networks: 0.3 to 1).  A sample's mark depends on its own rows only, so
// that its results do not depend on which samples share its tile or its unit.
//
// Roles: warps 0-11 epilogue (TMEM lane quarter w % 4, column part w / 4), warp 12 MMA issue,
// warps 13-15 weight producers.  Every wait is bounded; on timeout the kernel records
// TSDFS_DEV_TIMEOUT, drains its own copies and MMAs, frees TMEM and returns.
#include "tc_common.cuh"
#include "mlp_f32.cuh"

namespace tsdfs {

namespace {

constexpr int kTile = 32;             // samples per tile (four rows each)
constexpr int kTileV = 128;           // VALUE: samples per tile (one row each)
constexpr int kEpi = 12;              // epilogue warps: 4 lane quarters x 3 column parts
constexpr int kParts = 3;
constexpr int kMma = 12;              // MMA warp
constexpr int kStages = 2;
constexpr int kProd = 3;               // weight producers (16 warps in all leave 128 registers a thread)
constexpr int kItemParts = 2;          // copies of an item (hi and lo), each by the next producer in turn
// A producer waits for the release of the item kStages before its own by a parity, so the release before that
// one must be behind it: its last part was kProd parts ago, and it waited then for a release at most kStages
// items further back.  That also takes the MMA warp to release the stages in the items' order.
static_assert(kProd <= kItemParts * kStages, "a producer would wait a phase ahead of its stage");
constexpr int kThr = 32 * (kMma + 1 + kProd);
constexpr int kPh = 128;              // outputs per phase
constexpr int kGrp = 6;               // 8-column groups of a phase per part, at most
constexpr uint32_t kPartBytes = 64 * 1024;                 // 128 rows x 256 16-bit columns
constexpr uint32_t kStageBytes = 2 * kPh * kKChunk * 2;    // hi and lo of one item
constexpr int kUnit = 4;              // tiles per pass of the colour layers
constexpr float kUp = 32.0f;          // operand scale
constexpr float kLoUp = 2048.0f;      // further scale of the low part
constexpr float kDown = 1.0f / (kUp * kUp), kLoDown = 1.0f / kLoUp;
constexpr float kLimit = 2000.0f;     // largest operand the high part is trusted with
constexpr float kBias0 = 1.7e-8f, kBias1 = 1.58e-8f;   // what a main sum of n MMAs lacks: kBias0 + n kBias1
constexpr float kMinGrad = 1e-4f;
constexpr float kFloor = 1.0f / (16384.0f * kUp);   // 1.9e-6: the scaled high part of less is subnormal
constexpr int kMaxCtas = 192;         // CTAs that the workspace sizes have a place to park for
constexpr float kRsqrt2 = 0.70710678118654752f;

template <int ARCH> struct FArch {
    using A = Arch<ARCH>;
    static constexpr int LS = A::kSdfLayers;
    static constexpr int NL = A::kSdfLayers + A::kRgbLayers;
    static constexpr int kX = 3 + A::kDirEnc + 3;    // x~, direction encoding, unit normal
    static constexpr int kXp = pad16(kX);
    static constexpr int kF = A::kFeat;
    static constexpr int kFp = pad16(kF);
    __host__ __device__ static constexpr Layer layer(int L) { return L < LS ? A::sdf(L) : A::rgb(L - LS); }
    // layers with MMAs: all but the colour output; the SDF output's are the features only.
    // Operand columns in the main buffers (the colour input: its features), then the rest in its
    // own chunk; outputs padded to 16
    __host__ __device__ static constexpr int k_main(int L) { return L == LS ? kFp : pad16(layer(L).in); }
    __host__ __device__ static constexpr int n_pad(int L) { return L == LS - 1 ? kFp : pad16(layer(L).out); }
    __host__ __device__ static constexpr int main_chunks(int L) { return (k_main(L) + kKChunk - 1) / kKChunk; }
    __host__ __device__ static constexpr int chunks(int L) { return main_chunks(L) + (L == LS ? 1 : 0); }
    __host__ __device__ static constexpr int chunk_k(int L, int c) {
        return c == main_chunks(L) ? kXp : (k_main(L) - c * kKChunk < kKChunk ? k_main(L) - c * kKChunk : kKChunk);
    }
    __host__ __device__ static constexpr int phases(int L) { return (n_pad(L) + kPh - 1) / kPh; }
    __host__ __device__ static constexpr int phase_n(int L, int p) {
        return n_pad(L) - p * kPh < kPh ? n_pad(L) - p * kPh : kPh;
    }
    __host__ __device__ static constexpr int64_t layer_bytes(int L) {
        return (int64_t)n_pad(L) * (k_main(L) + (L == LS ? kXp : 0)) * 4;
    }
    __host__ __device__ static constexpr int64_t layer_base(int L) {
        int64_t o = 0;
        for (int l = 0; l < L; ++l) o += layer_bytes(l);
        return o;
    }
    __host__ __device__ static constexpr int64_t packed_bytes() { return layer_base(NL - 1); }
    __host__ __device__ static constexpr int items(int L0, int L1) {
        int n = 0;
        for (int L = L0; L < L1; ++L) n += phases(L) * chunks(L);
        return n;
    }
    __host__ __device__ static constexpr int bias_base(int L) {
        int o = 0;
        for (int l = 0; l < L; ++l) o += n_pad(l);
        return o;
    }
    __host__ __device__ static constexpr int64_t param_offset(int L) {
        return L < LS ? sdf_layer_offset<ARCH>(L) : rgb_layer_offset<ARCH>(L - LS);
    }
    // layer L's source row of padded output n, -1: padding
    __host__ __device__ static constexpr int src_row(int L, int n) {
        if (L == LS - 1) return n < kF ? n + 1 : -1;
        return n < layer(L).out ? n : -1;
    }
    // layer L's source column of padded input k (the colour input: features first), -1: padding
    __host__ __device__ static constexpr int src_col(int L, int k) {
        if (L == LS) return k < kF ? kX + k : (k >= kFp && k - kFp < kX ? k - kFp : -1);
        return k < layer(L).in ? k : -1;
    }
    template <bool VALUE> __host__ __device__ static constexpr int mma_layers() { return VALUE ? LS - 1 : NL - 1; }
    template <bool VALUE> __host__ __device__ static constexpr uint32_t table_floats() {
        return VALUE ? kTileV * (4 + 6 * A::kPeSdf) : kTile * (8 + 6 * (A::kPeSdf + A::kPeDir));
    }
    static constexpr int kChecked = NL - 2 - LS;   // colour layers whose outputs become operands
    // net_0's weights and partial sums (3 parts x 128 rows), the samples' marks; the record's SDF half,
    // the colour output's weights and partial sums (3 parts x 3 colours x 128 rows), the floor's checks
    static constexpr int kW0 = pad16(A::sdf(LS - 1).in), kWc = pad16(A::rgb(A::kRgbLayers - 1).in);
    template <bool VALUE> __host__ __device__ static constexpr uint32_t scratch_floats() {
        return kW0 + kParts * 128 + 32 + (VALUE ? 0 : kTile * 8 + 3 * kWc + kParts * 3 * 128 + (kTile + kChecked * 128) / 4);
    }
    // items of a tile's SDF layers, and of a unit's colour layers (the first one's phases take one
    // more each, the operand columns beyond the features)
    template <bool VALUE> __host__ __device__ static constexpr int sdf_items() { return items(0, VALUE ? LS - 1 : LS); }
    template <bool VALUE> __host__ __device__ static constexpr int n_items() {
        return VALUE ? sdf_items<true>() : items(0, NL - 1) + phases(LS);
    }
    // the parked colour inputs of a unit: the features' operand image (hi, lo), then the others'
    static constexpr uint32_t kParkF = 16u * (kFp / 8) * 128u, kParkX = 16u * (kXp / 8) * 128u;
    __host__ __device__ static constexpr size_t park_bytes() { return 2 * (size_t)(kParkF + kParkX); }
    template <bool VALUE> __host__ __device__ static constexpr uint32_t bias_floats() {
        return bias_base(mma_layers<VALUE>());
    }
    template <bool VALUE> __host__ __device__ static constexpr size_t smem_bytes() {
        return 2 * (size_t)kPartBytes + kStages * (size_t)kStageBytes + 4u * bias_floats<VALUE>() +
               4u * table_floats<VALUE>() + 4u * scratch_floats<VALUE>() + 32u * n_items<VALUE>() + 128;
    }
};

// one weight item as the MMA warp and the producers use it
struct __align__(16) Item {
    uint32_t off;      // of the hi part in the packed weights (the lo part follows)
    uint32_t bytes;    // of one part
    uint32_t a;        // operand offset of its first K step (hi part)
    uint32_t a_sbo;    // operand row-group stride
    uint32_t b_sbo;
    uint32_t idesc;
    uint16_t steps;    // K steps of 16
    uint16_t n;        // outputs
    uint16_t pad;
    uint16_t edge;     // bit 0: first item of a phase, bit 1: last, bit 2 / 3: its operand's columns below /
                       // from 128 are awaited first, bit 4: the parked features are, bit 5: an operand item
                       // (parked columns, no MMAs), bit 6: its operand is the item before
};
static_assert(sizeof(Item) == 32, "item record");

struct F32Params {
    const uint8_t* packed;
    const float* sdf_w;
    const float* rgb_w;
    float center[3];
    float inv_scale, scale, beta;
    SampleSource src;
    SampleRec* rec;      // full evaluation
    float* f_out;        // VALUE
    uint32_t* redo;      // set when a tile is marked
    uint8_t* park;       // FArch::park_bytes() per CTA
    uint32_t* status;
    uint32_t spin;
    int withhold;
};

__device__ __forceinline__ void wait_ld16(float (&a)[8], float (&b)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+f"(a[4]), "+f"(a[5]), "+f"(a[6]), "+f"(a[7]),
                   "+f"(b[0]), "+f"(b[1]), "+f"(b[2]), "+f"(b[3]), "+f"(b[4]), "+f"(b[5]), "+f"(b[6]), "+f"(b[7])
                 :
                 : "memory");
}
// global-memory writes of this thread before bulk copies that read them
__device__ __forceinline__ void fence_async_global() { asm volatile("fence.proxy.async;" ::: "memory"); }
// the two FP16 parts of a pair of FP32 operands times kUp (see the head of the file)
__device__ __forceinline__ void split_f32(float a, float b, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn((a - f.x) * kLoUp, (b - f.y) * kLoUp);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

__device__ __forceinline__ __half2 from_bits(uint32_t u) { return *reinterpret_cast<const __half2*>(&u); }

// softplus_beta(z) = max(z, 0) + log(1 + e^{-beta |z|}) / beta and its slope sigma(beta z).  The
// fast exponential and logarithm measure the same errors in f and grad f as expf and an FP32
// series for the logarithm (|grad f| 6.3e-8 off through the tiny networks either way).
__device__ __forceinline__ void softplus_slope_f32(float z, float beta, float inv_beta, float& h, float& sg) {
    const float u = beta * z;
    const float e = __expf(-fabsf(u)), d = 1.0f + e;
    const float r = __fdividef(1.0f, d);
    sg = u >= 0.0f ? r : e * r;
    h = fmaf(__logf(d), inv_beta, z < 0.0f ? 0.0f : z);
}

// max(x, 0) that keeps a NaN (so that it is noticed)
__device__ __forceinline__ float relu_nan(float x) { return x < 0.0f ? 0.0f : x; }

template <int ARCH, bool VALUE>
__global__ void __launch_bounds__(kThr, 1) k_mlp_f32(F32Params p) {
    using F = FArch<ARCH>;
    using A = Arch<ARCH>;
    constexpr int LS = F::LS, NLr = F::template mma_layers<VALUE>();
    constexpr int NT = F::template n_items<VALUE>();
    constexpr int TS = VALUE ? kTileV : kTile;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* a_hi = smem;
    uint8_t* a_lo = smem + kPartBytes;
    uint8_t* ring = smem + 2 * kPartBytes;
    float* s_bias = reinterpret_cast<float*>(ring + kStages * kStageBytes);
    float* s_x = s_bias + F::template bias_floats<VALUE>();
    constexpr int kXRow = VALUE ? 4 : 8;       // x~ (3), [direction (3), t, delta]
    float* s_pe = s_x + TS * kXRow;            // sin, cos of 2^oct x~_a
    float* s_pd = s_pe + TS * A::kPeSdf * 6;   // of the direction
    float* s_w0 = s_x + F::template table_floats<VALUE>();
    float* s_dot = s_w0 + F::kW0;                  // [part][row]
    volatile uint8_t* s_bad = reinterpret_cast<volatile uint8_t*>(s_dot + kParts * 128);   // [tile of the unit][sample]
    float* s_out = s_dot + kParts * 128 + 32;      // [sample][8]
    float* s_wc = s_out + kTile * 8;               // [colour][input]
    float* s_cdot = s_wc + 3 * F::kWc;             // [part][colour][row]
    // whether the tangents of each sample of the tile reach the floor in every layer, and the activations of
    // each sample of the unit in each colour layer
    volatile uint8_t* s_tan = reinterpret_cast<volatile uint8_t*>(s_cdot + kParts * 3 * 128);
    volatile uint8_t* s_act = s_tan + kTile;       // [colour layer][tile of the unit][sample]
    Item* items = reinterpret_cast<Item*>(s_w0 + F::template scratch_floats<VALUE>());
    uint64_t* bars = reinterpret_cast<uint64_t*>(items + NT);
    // bars: full[2], empty[2], acc[2], drained[2], operand[2], epi, end, parked, back
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 14);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile uint32_t* s_low = tmem_slot + 2;   // a layer's weights are all below the floor
    const uint32_t bar_full = smem_u32(bars), bar_empty = smem_u32(bars + kStages);
    const uint32_t bar_acc = smem_u32(bars + 4), bar_drained = smem_u32(bars + 6), bar_op = smem_u32(bars + 8),
                   bar_epi = smem_u32(bars + 10), bar_end = smem_u32(bars + 11), bar_park = smem_u32(bars + 12),
                   bar_back = smem_u32(bars + 13);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    const int64_t total = sample_total(p.src);
    if (total > p.src.capacity) {
        if (blockIdx.x == 0 && threadIdx.x == 0) set_status(p.status, TSDFS_DEV_SAMPLES_OVERFLOW);
        return;
    }
    const int64_t n_tiles = (total + TS - 1) / TS;
    if ((int64_t)blockIdx.x >= n_tiles) return;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(bar_full + 8 * i, kItemParts);
            mbar_init(bar_empty + 8 * i, 1);
            mbar_init(bar_acc + 8 * i, 1);
            mbar_init(bar_drained + 8 * i, kEpi);
            mbar_init(bar_op + 8 * i, kEpi);
        }
        mbar_init(bar_epi, kEpi);
        mbar_init(bar_end, 1);
        mbar_init(bar_park, kEpi);
        mbar_init(bar_back, 1);
        *abort_flag = 0;
        uint32_t low = 0;
        for (int L = 0; L < NLr; ++L) low |= __ldg(p.redo + kLowWord + L);
        *s_low = low;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the items in order: layers, phases, chunks; a thread writes one layer's
    if (threadIdx.x < NLr) {
        const int L = threadIdx.x;
        uint32_t off = (uint32_t)F::layer_base(L);
        int j = F::items(0, L) + (L > LS ? F::phases(LS) : 0);
        const uint32_t sbo = (uint32_t)(F::k_main(L) / 8) * 128u;
        for (int ph = 0; ph < F::phases(L); ++ph) {
            const int n = F::phase_n(L, ph);
            for (int c = 0; c < F::chunks(L); ++c) {
                Item it;
                const int kc = F::chunk_k(L, c);
                const bool extra = c == F::main_chunks(L);   // the colour input's columns beyond the features
                it.off = off;
                it.bytes = (uint32_t)(n * kc * 2);
                off += 2 * it.bytes;
                it.a = extra ? 0u : (uint32_t)(c * (kKChunk / 8)) * 128u;
                it.a_sbo = extra ? (uint32_t)(F::kXp / 8) * 128u : sbo;
                it.b_sbo = (uint32_t)(kc / 8) * 128u;
                it.idesc = idesc_mma<true>(128, n);
                it.steps = (uint16_t)(kc / 16);
                it.n = (uint16_t)n;
                it.pad = 0;
                const bool back = L == LS && ph == 0 && c == 0;
                it.edge = (uint16_t)((c == 0 ? 1 : 0) | (c + 1 == F::chunks(L) ? 2 : 0) | (L != LS && ph == 0 && c == 0 ? 4 : 0) |
                                     (L != LS && ph == 0 && c * kKChunk == kPh ? 8 : 0) | (back ? 16 : 0) | (extra ? 64 : 0));
                if (extra) {
                    Item x = it;
                    x.off = 2 * F::kParkF;
                    x.bytes = F::kParkX;
                    x.edge = 32;
                    items[j++] = x;
                }
                items[j++] = it;
            }
        }
    }
    static_for<0, NLr>([&](auto lc) {
        constexpr int L = decltype(lc)::value;
        constexpr Layer ly = F::layer(L);
        const float* b = (L < LS ? p.sdf_w : p.rgb_w) + F::param_offset(L) + (int64_t)ly.out * ly.in;
        for (int i = threadIdx.x; i < F::n_pad(L); i += kThr) {
            const int r = F::src_row(L, i);
            s_bias[F::bias_base(L) + i] = r >= 0 ? __ldg(b + r) : 0.0f;
        }
    });
    for (int i = threadIdx.x; i < 128; i += kThr) s_bad[i] = 0;
    if constexpr (!VALUE)
        for (int i = threadIdx.x; i < kTile + F::kChecked * 128; i += kThr) s_tan[i] = 0;
    for (int i = threadIdx.x; i < F::kW0; i += kThr) {
        constexpr int K = A::sdf(LS - 1).in;
        s_w0[i] = i < K ? __ldg(p.sdf_w + F::param_offset(LS - 1) + i) : 0.0f;
    }
    if constexpr (!VALUE) {
        constexpr int K = A::rgb(A::kRgbLayers - 1).in;
        for (int i = threadIdx.x; i < 3 * F::kWc; i += kThr) {
            const int k = i % F::kWc;
            s_wc[i] = k < K ? __ldg(p.rgb_w + F::param_offset(F::NL - 1) + (i / F::kWc) * K + k) : 0.0f;
        }
    }
    if (warp == kMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // this CTA's tiles: blockIdx.x + k gridDim.x, k < mine; units of kUnit of them (VALUE: one)
    const int64_t mine = (n_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x;
    constexpr int kU = VALUE ? 1 : kUnit, NS = F::template sdf_items<VALUE>();
    auto tile_of = [&](int64_t k) { return blockIdx.x + k * gridDim.x; };
    uint8_t* park = VALUE ? nullptr : p.park + (size_t)blockIdx.x * F::park_bytes();

    if (warp > kMma) {
        // ---------------------------------------- producers: the items' parts in turn
        if (lane == 0) {
            int64_t last = -1, g = 0;       // the last item this thread copied a part of, the item in hand
            int turn = warp - kMma - 1;     // parts until this thread's next one
            uint32_t parked = 0;            // units up to the one in hand
            bool ok = true;
            auto item = [&](int j) {
                const bool operand = (items[j].edge & 32u) != 0;
                for (uint32_t part = 0; part < kItemParts; ++part, --turn) {
                    if (turn != 0) continue;
                    turn = kProd;
                    const uint32_t stage = (uint32_t)g & 1u;
                    if (p.withhold >= 0 && g >= p.withhold) { ok = false; return; }   // test-only: never issued
                    const uint32_t off = items[j].off, bytes = items[j].bytes;
                    if (operand && !mbar_wait(bar_park, (parked - 1) & 1u, abort_flag, p.spin)) { ok = false; return; }
                    if (!mbar_wait(bar_empty + 8 * stage, ((uint32_t)(g >> 1) & 1u) ^ 1u, abort_flag, p.spin)) { ok = false; return; }
                    mbar_expect_tx(bar_full + 8 * stage, bytes);
                    bulk_g2s(smem_u32(ring) + stage * kStageBytes + part * bytes, (operand ? park : p.packed) + off + part * bytes,
                             bytes, bar_full + 8 * stage);
                    last = g;
                }
                ++g;
            };
            for (int64_t k = 0; k < mine && ok; k += kU) {
                const int nt = mine - k < kU ? (int)(mine - k) : kU;
                for (int i = 0; i < nt && ok; ++i)
                    for (int j = 0; j < NS && ok; ++j) item(j);
                ++parked;
                for (int j = NS; j < NT && ok; ++j) item(j);
            }
            if (!ok && last >= 0) {
                // a copy of this thread may be in flight: its phase completes once the other part is
                // there too, so wait (bounded) before the CTA's shared memory goes away
                for (uint32_t it = 0; it < (1u << 20) && !mbar_try(bar_full + 8 * ((uint32_t)last & 1u), (uint32_t)(last >> 1) & 1u); ++it) {
                }
            }
        }
    } else if (warp == kMma) {
        // ---------------------------------------- MMA issue (the warp converged, one lane elected)
        const uint32_t el = elect_one();
        const uint32_t ah0 = smem_u32(a_hi), al0 = smem_u32(a_lo), r0 = smem_u32(ring);
        uint32_t g = 0, ph = 0, op_a = 0, op_b = 0;   // items, phases, waits for either half of an operand
        bool ok = true;
        auto wait = [&](uint32_t bar, uint32_t parity) {
            return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, p.spin));
        };
        uint32_t back = 0;
        auto run = [&](int j0, int j1) {
            for (int j = j0; j < j1; ++j, ++g) {
                const Item it = items[j];
                const uint32_t stage = g & 1u;
                if (it.edge & 32u) continue;   // an operand: the next item waits for it
                if ((it.edge & 4u) && !wait(bar_op, op_a++ & 1u)) return false;
                if ((it.edge & 8u) && !wait(bar_op + 8, op_b++ & 1u)) return false;
                if ((it.edge & 16u) && !wait(bar_back, back++ & 1u)) return false;
                // the buffer's previous phase has been read
                if ((it.edge & 1u) && ph >= 2 && !wait(bar_drained + 8 * (ph & 1u), ((ph >> 1) - 1) & 1u)) return false;
                if ((it.edge & 64u) && !wait(bar_full + 8 * (stage ^ 1u), ((g - 1) >> 1) & 1u)) return false;
                if (!wait(bar_full + 8 * stage, (g >> 1) & 1u)) return false;
                tc_fence_after();
                const uint32_t b = r0 + stage * kStageBytes;
                uint64_t bh = mdesc(b, 128, it.b_sbo);
                const uint32_t ax = r0 + (stage ^ 1u) * kStageBytes;
                uint64_t ah = mdesc(it.edge & 64u ? ax : ah0 + it.a, 128, it.a_sbo);
                uint64_t al = mdesc(it.edge & 64u ? ax + F::kParkX : al0 + it.a, 128, it.a_sbo);
                const uint32_t d_main = tmem + (ph & 1u) * (2 * kPh), d_corr = d_main + it.n;
                const uint32_t idesc2 = idesc_mma<true>(128, 2 * it.n);   // both parts of the weights
                const uint32_t acc = it.edge & 1u ? 0u : 1u;
                auto step = [&](int k) {
                    mma_el(el, d_main, ah + 16 * k, bh + 16 * k, idesc2, k > 0 ? 1u : acc);
                    mma_el(el, d_corr, al + 16 * k, bh + 16 * k, it.idesc, 1u);
                };
                if (it.steps == kKChunk / 16) static_for<0, kKChunk / 16>([&](auto k) { step(decltype(k)::value); });
                else
                    for (int k = 0; k < it.steps; ++k) step(k);
                if (it.edge & 64u) commit_el(el, bar_empty + 8 * (stage ^ 1u));   // the operand item is the earlier one
                commit_el(el, bar_empty + 8 * stage);
                if (it.edge & 2u) commit_el(el, bar_acc + 8 * (ph++ & 1u));
            }
            return true;
        };
        for (int64_t k = 0; k < mine && ok; k += kU) {
            const int nt = mine - k < kU ? (int)(mine - k) : kU;
            for (int i = 0; i < nt && ok; ++i) ok = run(0, NS);
            if (ok) ok = run(NS, NT);
        }
        if (!ok && el) {
            mma_commit(bar_end);
            for (uint32_t it = 0; it < kMaxSpin && !mbar_try(bar_end, 0); ++it) {
            }
        }
    } else {
        // ---------------------------------------- epilogue
        const int q = warp & 3, pt = warp >> 2;
        const int sq = lane >> 2, fc = 2 * (lane & 3);
        const uint32_t lq = (uint32_t)(32 * q) << 16, lq16 = (uint32_t)(32 * q + 16) << 16;
        const float inv_beta = 1.0f / p.beta;
        const float b0 = __ldg(p.sdf_w + F::param_offset(LS - 1) + (int64_t)F::layer(LS - 1).out * F::layer(LS - 1).in);
        const int et = threadIdx.x;
        uint32_t phs = 0, epi_ph = 0, backs = 0;   // phases waited for, epilogue barriers, units fetched back
        uint32_t buf = 0, cor = 0;                // TMEM columns of the phase in hand: main, correction
        // largest |operand| (scaled high parts) or NaN of the sample this thread works for; VALUE: of each of
        // its four rows' samples
        constexpr int kOwn = VALUE ? 4 : 1;
        __half2 big[kOwn];
#pragma unroll
        for (int r = 0; r < kOwn; ++r) big[r] = __float2half2_rn(0.0f);
        // full evaluation: the same of its tangents in the layer in hand, and the smallest such of its layers
        constexpr uint32_t kInf2 = 0x7c007c00u;
        __half2 tang = __float2half2_rn(0.0f), least = from_bits(kInf2);
        bool ok = true;
        auto epi_sync = [&]() -> bool {
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_epi);
            const bool w = mbar_wait(bar_epi, epi_ph & 1u, abort_flag, p.spin);
            ++epi_ph;
            return __all_sync(0xffffffffu, w);
        };
        auto wait_acc = [&](int n) -> bool {       // n: the phase's outputs
            const uint32_t b = phs & 1u;
            const bool w = __all_sync(0xffffffffu, mbar_wait(bar_acc + 8 * b, (phs >> 1) & 1u, abort_flag, p.spin));
            ++phs;
            buf = tmem + b * (2 * kPh);
            cor = buf + n;
            tc_fence_after();
            return w;
        };
        // the phase in hand has been read by this warp
        auto drained = [&]() {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_drained + 8 * ((phs - 1) & 1u));
        };
        // this warp's share of the next operand's columns below (0) or from (1) 128 is stored
        auto operand_done = [&](int half) {
            fence_proxy_async();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_op + 8 * half);
        };
        // a phase's raw accumulators of one 8-column group: row groups 0-3 of this thread, two columns
        auto issue4 = [&](int c, float (&m)[8], float (&cr)[8]) {
            tmem_ld16x256_x1(buf + lq + c, m);
            tmem_ld16x256_x1(buf + lq16 + c, m + 4);
            tmem_ld16x256_x1(cor + lq + c, cr);
            tmem_ld16x256_x1(cor + lq16 + c, cr + 4);
        };
        // rows 0-15 only: the value rows' registers are 0 and 1
        auto issue1 = [&](int c, float (&m)[4], float (&cr)[4]) {
            tmem_ld16x256_x1(buf + lq + c, m);
            tmem_ld16x256_x1(cor + lq + c, cr);
        };
        // row i of the lane quarter (stmatrix: lane i addresses row i) at column 0
        auto row_at = [&](uint8_t* base, int r, int pitch) { return smem_u32(base) + a_off(32 * q + r, 0, pitch); };
        // sample (VALUE: its row) that row group r of this thread belongs to
        auto sample_of = [&](int r) { return VALUE ? 32 * q + 8 * r + sq : 8 * q + sq; };
        auto enc = [&](int r, int j) {
            const int s = sample_of(r);
            return enc_tab(s_x + s * kXRow, s_pe + s * A::kPeSdf * 6, A::kPeSdf, j, VALUE ? 0 : r);
        };
        auto split = [&](float a, float b, uint32_t& hi, uint32_t& lo, __half2& most) {
            split_f32(a, b, hi, lo);
            most = __hmax2_nan(most, __habs2(*reinterpret_cast<const __half2*>(&hi)));
        };
        // split the four row groups' column pairs v (operands times kUp)
        auto split4 = [&](const float (&v)[8], uint32_t (&o)[8]) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                if constexpr (VALUE) split(v[2 * r], v[2 * r + 1], o[r], o[4 + r], big[r]);
                else split(v[2 * r], v[2 * r + 1], o[r], o[4 + r], r > 0 ? tang : big[0]);
            }
        };
        // the tangents since the last call join what out_of_range tells of
        auto fold_tangents = [&]() {
            big[0] = __hmax2_nan(big[0], tang);
            tang = __float2half2_rn(0.0f);
        };
        // whether one of two largest high parts is above the floor: a normal number
        auto reaches = [](__half2 most) { return (*reinterpret_cast<const uint32_t*>(&most) & kInf2) != 0; };
        // whether a value since the last call was out of the parts' range
        auto out_of_range = [&](__half2& most) {
            const float2 m = __half22float2(most);
            most = __float2half2_rn(0.0f);
            return !(fmaxf(m.x, m.y) < kUp * kLimit && m.x == m.x && m.y == m.y);
        };
        auto store4 = [&](uint32_t rh, uint32_t rl, int c, const uint32_t (&o)[8]) {
            const uint32_t co = (uint32_t)(c >> 3) * 128u;
            stmatrix4(rh + co, o[0], o[1], o[2], o[3]);
            stmatrix4(rl + co, o[4], o[5], o[6], o[7]);
        };
        // the tile's table: x~ (and direction, t, delta), then sin / cos of the encodings' octaves
        auto build_table = [&](int64_t tile) -> bool {
            if (et < TS) {
                const int64_t g = tile * TS + et;
                float t = 0.0f, dl = 0.0f, xs[3] = {0.0f, 0.0f, 0.0f}, ds[3] = {0.0f, 0.0f, 0.0f};
                if (g < total) {
                    int64_t ray;
                    if (p.src.mode == kUniform) {
                        ray = p.src.sample_ray ? (int64_t)__ldg(p.src.sample_ray + g) : find_ray(p.src.offsets, p.src.n_rays, g);
                        const int32_t o0 = __ldg(p.src.offsets + ray), o1 = __ldg(p.src.offsets + ray + 1);
                        const float tn = __ldg(p.src.t_n + ray), tf = __ldg(p.src.t_f + ray);
                        dl = (tf - tn) / (float)(o1 - o0);
                        t = tn + ((float)(g - o0) + 0.5f) * dl;
                    } else {
                        ray = explicit_ray(p.src, g);
                        t = __ldg(p.src.t + g);
                        if constexpr (!VALUE) dl = __ldg(p.src.delta + g);
                    }
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        ds[a] = __ldg(p.src.ray_d + 3 * ray + a);
                        const float x = __ldg(p.src.ray_o + 3 * ray + a) + t * ds[a];
                        xs[a] = (x - p.center[a]) * p.inv_scale;
                    }
                }
                float* sx = s_x + et * kXRow;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    sx[a] = xs[a];
                    if constexpr (!VALUE) sx[3 + a] = ds[a];
                }
                if constexpr (!VALUE) {
                    sx[6] = t;
                    sx[7] = dl;
                }
            }
            if (!epi_sync()) return false;
            constexpr int nd = VALUE ? 0 : A::kPeDir, per = 3 * (A::kPeSdf + nd);
            constexpr int div = per > 0 ? per : 1;
            for (int e = et; e < TS * per; e += kEpi * 32) {
                const int s = e / div, k = e % div;
                const bool dir = k >= 3 * A::kPeSdf;
                const int i = dir ? k - 3 * A::kPeSdf : k;    // octave * 3 + axis
                float sn, cs;
                sincosf((float)(1 << (i / 3)) * s_x[s * kXRow + (dir ? 3 : 0) + i % 3], &sn, &cs);
                float* dst = (dir ? s_pd + s * A::kPeDir * 6 : s_pe + s * A::kPeSdf * 6) + 2 * i;
                dst[0] = sn;
                dst[1] = cs;
            }
            return epi_sync();
        };
        auto write_input0 = [&]() {
            constexpr int K0 = F::k_main(0);
            const uint32_t rh = row_at(a_hi, lane, K0), rl = row_at(a_lo, lane, K0);
            for (int gr = pt; gr < K0 / 8; gr += kParts) {
                float v[8];
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int j = 8 * gr + fc + e;
                        v[2 * r + e] = j < A::kEnc ? enc(r, j) * kUp : 0.0f;
                    }
                uint32_t o[8];
                split4(v, o);
                store4(rh, rl, 8 * gr, o);
            }
            if constexpr (!VALUE) fold_tangents();
            operand_done(0);
        };

        // a phase's 8-column groups of this part, two at a time.  What a group takes is a chain of some
        // 40 dependent instructions, and three warps to a scheduler do not hide it: two groups wholly
        // below n_fast go through act(c, z, o) as one straight run of code that interleaves, and only
        // the others branch per column, through edge(c, z, o).  (One group at a time, with the branches:
        // 1330 cycles a group and warp.)  put(i, c, o) takes the results; accumulators end at n_acc
        // (zero sums beyond), groups at n_all.
        auto groups = [&](float share, int n_fast, int n_acc, int n_all, auto act, auto edge, auto put) {
#pragma unroll
            for (int i = 0; i < kGrp; i += 2) {
                const int c0 = 8 * (pt + i * kParts), c1 = c0 + 8 * kParts;
                if (c0 >= n_all) continue;
                float z0[8], z1[8], r0[8], r1[8];
                uint32_t o0[8], o1[8];
                const bool ld0 = c0 < n_acc, ld1 = c1 < n_acc;
                if (ld0) issue4(c0, z0, r0);
                if (ld1) issue4(c1, z1, r1);
                wait_ld16(z0, r0);
                wait_ld16(z1, r1);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    z0[k] = fmaf(z0[k], share, fmaf(r0[k], kLoDown, z0[k]));
                    z1[k] = fmaf(z1[k], share, fmaf(r1[k], kLoDown, z1[k]));
                }
                if (c1 + 8 <= n_fast) {
                    act(c0, z0, o0);
                    act(c1, z1, o1);
                    put(i, c0, o0);
                    put(i + 1, c1, o1);
                } else {
                    if (c0 + 8 <= n_fast) act(c0, z0, o0);
                    else {
                        if (!ld0) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) z0[k] = 0.0f;
                        }
                        edge(c0, z0, o0);
                    }
                    put(i, c0, o0);
                    if (c1 < n_all) {
                        if (!ld1) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) z1[k] = 0.0f;
                        }
                        edge(c1, z1, o1);
                        put(i + 1, c1, o1);
                    }
                }
            }
        };
        ok = build_table(blockIdx.x);
        if (ok) write_input0();
        for (int64_t kt = 0; kt < mine && ok; ++kt) {
            const int64_t tile = tile_of(kt);
            const int slot = (int)(kt % kU);                        // of its unit
            const bool unit_end = slot == kU - 1 || kt + 1 == mine;
            const float* bias = s_bias;
            for (int L = 0; L < (unit_end ? NLr : (NLr < LS ? NLr : LS)) && ok; bias += F::n_pad(L), ++L) {
                // a single K step (the 3 raw coordinates and their one-hot derivatives) is exact or nearly so
                const int n_mma = (F::k_main(L) + (L == LS ? F::kXp : 0)) / 16;
                const float share = n_mma > 1 ? kBias0 + kBias1 * (float)n_mma : 0.0f;
                if (L < LS - 1) {
                    // ---- hidden SDF layer: softplus on value rows, its slope times the tangent rows ----
                    const int N = F::layer(L).out, Np = F::n_pad(L), Kn = F::k_main(L + 1);
                    const bool skip = L + 1 == A::kSkip;
                    const bool last = L == LS - 2;             // net_0's dot products are taken here
                    const bool store = !(VALUE && last);
                    float dot[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    const float sc = skip ? kRsqrt2 : 1.0f;
                    const uint32_t rh = row_at(a_hi, lane, Kn), rl = row_at(a_lo, lane, Kn);
                    // accumulator sums z of operand columns c .. c + 7 -> both parts of the next operand; the
                    // scales are powers of two (but sc), so where they are applied changes no bit
                    auto act = [&](int c, const float (&z)[8], uint32_t (&o)[8]) {
                        float v[8];
                        const float2 b = *reinterpret_cast<const float2*>(bias + c + fc);
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            float h, sg;
                            if constexpr (VALUE) {
#pragma unroll
                                for (int r = 0; r < 4; ++r) {
                                    softplus_slope_f32(fmaf(z[2 * r + e], kDown, e ? b.y : b.x), p.beta, inv_beta, h, sg);
                                    v[2 * r + e] = h * (sc * kUp);
                                }
                            } else {
                                softplus_slope_f32(fmaf(z[e], kDown, e ? b.y : b.x), p.beta, inv_beta, h, sg);
                                v[e] = h * (sc * kUp);
                                sg *= sc * kUp * kDown;
#pragma unroll
                                for (int r = 1; r < 4; ++r) v[2 * r + e] = sg * z[2 * r + e];
                            }
                        }
                        if (last) {
                            const float2 w = *reinterpret_cast<const float2*>(s_w0 + c + fc);
#pragma unroll
                            for (int r = 0; r < 4; ++r) dot[r] = fmaf(v[2 * r + 1], w.y, fmaf(v[2 * r], w.x, dot[r]));
                        }
                        split4(v, o);
                    };
                    // some of the columns are beyond the outputs: the skip input's encoding, or padding
                    auto edge = [&](int c, const float (&z)[8], uint32_t (&o)[8]) {
                        float v[8];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int col = c + fc + e;
                            if (col < N) {
                                const float b = bias[col];
                                float h, sg;
#pragma unroll
                                for (int r = 0; r < (VALUE ? 4 : 1); ++r) {
                                    softplus_slope_f32(fmaf(z[2 * r + e], kDown, b), p.beta, inv_beta, h, sg);
                                    v[2 * r + e] = h * (sc * kUp);
                                }
                                if constexpr (!VALUE) {
                                    sg *= sc * kUp * kDown;
#pragma unroll
                                    for (int r = 1; r < 4; ++r) v[2 * r + e] = sg * z[2 * r + e];
                                }
                                if (last) {
                                    const float w = s_w0[col];
#pragma unroll
                                    for (int r = 0; r < 4; ++r) dot[r] = fmaf(v[2 * r + e], w, dot[r]);
                                }
                            } else {
                                const bool in = skip && col - N < A::kEnc;
#pragma unroll
                                for (int r = 0; r < 4; ++r) v[2 * r + e] = in ? enc(r, col - N) * (sc * kUp) : 0.0f;
                            }
                        }
                        split4(v, o);
                    };
                    uint32_t held[kGrp][8];
                    const bool two = Np > kPh;
                    if (two) {
                        if (!wait_acc(kPh)) { ok = false; break; }
                        groups(share, kPh, kPh, kPh, act, edge, [&](int i, int, const uint32_t (&o)[8]) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) held[i][k] = o[k];
                        });
                        drained();
                    }
                    const int n0 = two ? kPh : 0;
                    if (!wait_acc(Np - n0)) { ok = false; break; }
                    if (two && store) {
#pragma unroll
                        for (int i = 0; i < kGrp; ++i)
                            if (pt + i * kParts < kPh / 8) store4(rh, rl, 8 * (pt + i * kParts), held[i]);
                        operand_done(0);
                    }
                    groups(share, N - n0, Np - n0, Kn - n0,
                           [&](int c, const float (&z)[8], uint32_t (&o)[8]) { act(n0 + c, z, o); },
                           [&](int c, const float (&z)[8], uint32_t (&o)[8]) { edge(n0 + c, z, o); },
                           [&](int, int c, const uint32_t (&o)[8]) {
                               if (store) store4(rh, rl, n0 + c, o);
                           });
                    drained();
                    if (store) operand_done(two ? 1 : 0);
                    if constexpr (!VALUE) {
                        // (the last layer's tangents are summed in FP32.)  One thread with a tangent above the floor
                        // in every layer will do
                        if (!last) {
                            least = __hmin2(least, tang);
                        } else {
                            if (reaches(least)) s_tan[sample_of(0)] = 1;
                            least = from_bits(kInf2);
                        }
                        fold_tangents();
                    }
                    if (last) {
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            dot[r] += __shfl_xor_sync(0xffffffffu, dot[r], 1);
                            dot[r] += __shfl_xor_sync(0xffffffffu, dot[r], 2);
                            if ((lane & 3) == 0) s_dot[pt * 128 + 32 * q + 8 * r + sq] = dot[r] * (1.0f / kUp);
                        }
                    }
                    if constexpr (VALUE) {
                        if (last) {
                            // the SDF values, and the next tile's input
#pragma unroll
                            for (int r = 0; r < 4; ++r)
                                if (out_of_range(big[r])) s_bad[sample_of(r)] = 1;
                            if (!epi_sync()) { ok = false; break; }
                            if (et < TS) {
                                const float f = p.scale * (s_dot[et] + s_dot[128 + et] + s_dot[256 + et] + b0);
                                const bool bad = *s_low != 0 || s_bad[et] != 0 || !(fabsf(f) < __int_as_float(0x7f800000));
                                s_bad[et] = 0;
                                if (tile * TS + et < total) {
                                    p.f_out[tile * TS + et] = bad ? __uint_as_float(kRedoBits) : f;
                                    if (bad) atomicExch(p.redo, 1u);
                                }
                            }
                            if (kt + 1 < mine) {
                                if (!build_table(tile_of(kt + 1))) { ok = false; break; }
                                write_input0();
                            }
                        }
                    }
                } else if (L == LS - 1) {
                    // ---- SDF output: the features; net_0 and its gradient from their dot products ----
                    if constexpr (!VALUE) {
                        constexpr int NF = F::phases(LS - 1);
                        // value row sq of quarter q goes to row group `slot` of it; a warp's 8 rows x 8
                        // columns are one core matrix, 128 bytes in lane order
                        uint8_t* pf = park + (4 * q + slot) * (F::kFp / 8) * 128 + 4 * lane;
#pragma unroll
                        for (int ph = 0; ph < NF; ++ph) {
                            if (!wait_acc(F::phase_n(LS - 1, ph))) { ok = false; break; }
                            constexpr int kAt = kGrp / 2;   // groups whose loads are in flight together
#pragma unroll
                            for (int i0 = 0; i0 < kGrp; i0 += kAt) {
                                float m[kAt][4], cr[kAt][4];
#pragma unroll
                                for (int i = 0; i < kAt; ++i) {
                                    const int c = 8 * (pt + (i0 + i) * kParts);
                                    if (c < F::phase_n(LS - 1, ph)) issue1(c, m[i], cr[i]);
                                }
#pragma unroll
                                for (int i = 0; i < kAt; ++i)
                                    asm volatile("tcgen05.wait::ld.sync.aligned;"
                                                 : "+f"(m[i][0]), "+f"(m[i][1]), "+f"(cr[i][0]), "+f"(cr[i][1])
                                                 :
                                                 : "memory");
#pragma unroll
                                for (int i = 0; i < kAt; ++i) {
                                    const int c = 8 * (pt + (i0 + i) * kParts);
                                    if (c >= F::phase_n(LS - 1, ph)) continue;
                                    float z[2];
#pragma unroll
                                    for (int e = 0; e < 2; ++e) {
                                        z[e] = fmaf(m[i][e], share, fmaf(cr[i][e], kLoDown, m[i][e]));
                                        z[e] = fmaf(z[e], kDown, bias[ph * kPh + c + fc + e]) * kUp;
                                    }
                                    uint32_t hi, lo;
                                    split(z[0], z[1], hi, lo, big[0]);
                                    uint32_t* at = reinterpret_cast<uint32_t*>(pf + (ph * kPh + c) / 8 * 128);
                                    at[0] = hi;
                                    at[F::kParkF / 4] = lo;
                                }
                            }
                            drained();
                            if (ph > 0) continue;
                            if (!epi_sync()) { ok = false; break; }
                            if (et < kTile) {
                                const int s = et, row = 32 * (s >> 3) + (s & 7);
                                float n0[4];
#pragma unroll
                                for (int r = 0; r < 4; ++r)
                                    n0[r] = s_dot[row + 8 * r] + s_dot[128 + row + 8 * r] + s_dot[256 + row + 8 * r];
                                const float f = p.scale * (n0[0] + b0), gx = n0[1], gy = n0[2], gz = n0[3];
                                const float gn = sqrtf(gx * gx + gy * gy + gz * gz);
                                const float inv = gn > 0.0f ? 1.0f / gn : 0.0f;
                                const float* sx = s_x + s * 8;
                                float* so = s_out + s * 8;
                                so[0] = gx * inv;
                                so[1] = gy * inv;
                                so[2] = gz * inv;
                                if (s_tan[s] == 0) s_bad[kTile * slot + s] = 1;
                                s_tan[s] = 0;
                                const int64_t g = tile * kTile + s;
                                if (g < total) {
                                    float4* R4 = reinterpret_cast<float4*>(p.rec + g);
                                    R4[0] = make_float4(f, gx * sx[3] + gy * sx[4] + gz * sx[5], sx[6], sx[7]);
                                    R4[2] = make_float4(so[0], so[1], so[2], 0.0f);
                                    p.rec[g].gnorm = gn;
                                    const float inf = __int_as_float(0x7f800000);
                                    if (!(gn >= kMinGrad && gn < inf) || !(fabsf(f) < inf)) s_bad[kTile * slot + s] = 1;
                                }
                            }
                        }
                        if (!ok) break;
                        // the tile's SDF operands and features (read and cleared by the unit's last thread for the
                        // sample, an epi_sync before this tile's first mark)
                        if (out_of_range(big[0])) s_bad[kTile * slot + sample_of(0)] = 1;
                        if (!epi_sync()) { ok = false; break; }
                        // x~, direction encoding, unit normal: one 8-column group of a sample per thread
                        if (et < kTile * (F::kXp / 8)) {
                            const int s = et / (F::kXp / 8), c = 8 * (et % (F::kXp / 8));
                            uint32_t o[8];
                            __half2 most = __float2half2_rn(0.0f);
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                float v[2];
#pragma unroll
                                for (int e = 0; e < 2; ++e) {
                                    const int j = c + 2 * k + e;
                                    v[e] = 0.0f;
                                    if (j < 3) v[e] = s_x[s * 8 + j];
                                    else if (j < 3 + A::kDirEnc)
                                        v[e] = enc_tab(s_x + s * 8 + 3, s_pd + s * A::kPeDir * 6, A::kPeDir, j - 3, 0);
                                    else if (j < F::kX) v[e] = s_out[s * 8 + j - 3 - A::kDirEnc];
                                }
                                split(v[0] * kUp, v[1] * kUp, o[k], o[4 + k], most);
                            }
                            if (out_of_range(most)) s_bad[kTile * slot + s] = 1;
                            uint8_t* at = park + 2 * F::kParkF + a_off(32 * (s >> 3) + 8 * slot + (s & 7), c, F::kXp);
                            *reinterpret_cast<uint4*>(at) = make_uint4(o[0], o[1], o[2], o[3]);
                            *reinterpret_cast<uint4*>(at + F::kParkX) = make_uint4(o[4], o[5], o[6], o[7]);
                        }
                        fence_async_global();
                        __syncwarp();
                        if (unit_end && lane == 0) mbar_arrive(bar_park);
                        if (!epi_sync()) { ok = false; break; }
                        if (unit_end && et == 0) {
                            // the unit's features as the operand (the SDF MMAs are complete)
                            fence_async_global();
                            mbar_expect_tx(bar_back, 2 * F::kParkF);
                            ++backs;
                            bulk_g2s(smem_u32(a_hi), park, F::kParkF, bar_back);
                            bulk_g2s(smem_u32(a_lo), park + F::kParkF, F::kParkF, bar_back);
                        }
                        // this tile's table is read no more: the next tile's (while the colour layers run, at
                        // a unit's end)
                        if (kt + 1 < mine && !build_table(tile_of(kt + 1))) { ok = false; break; }
                        if (!unit_end) write_input0();
                    }
                } else {
                    // ---- hidden colour layer: ReLU, all rows (row group j: tile j of the unit) ----
                    const int Np = F::n_pad(L);
                    const bool last = L == F::NL - 2;          // the colours' dot products are taken here
                    const uint32_t rh = row_at(a_hi, lane, Np), rl = row_at(a_lo, lane, Np);
                    float cd[3][4] = {};
                    __half2 most[4];                           // of each row group
#pragma unroll
                    for (int r = 0; r < 4; ++r) most[r] = __float2half2_rn(0.0f);
                    auto act = [&](int c, const float (&z)[8], uint32_t (&o)[8]) {
                        float v[8];
                        const float2 b = *reinterpret_cast<const float2*>(bias + c + fc);
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            v[2 * r] = relu_nan(fmaf(z[2 * r], kDown * kUp, b.x * kUp));
                            v[2 * r + 1] = relu_nan(fmaf(z[2 * r + 1], kDown * kUp, b.y * kUp));
                            // rows of tiles the unit does not have are nobody's
                            if (r > slot) v[2 * r] = v[2 * r + 1] = 0.0f;
                        }
                        if (last) {
#pragma unroll
                            for (int k = 0; k < 3; ++k) {
                                const float2 w = *reinterpret_cast<const float2*>(s_wc + k * F::kWc + c + fc);
#pragma unroll
                                for (int r = 0; r < 4; ++r) cd[k][r] = fmaf(v[2 * r + 1], w.y, fmaf(v[2 * r], w.x, cd[k][r]));
                            }
                        } else {
#pragma unroll
                            for (int r = 0; r < 4; ++r) split(v[2 * r], v[2 * r + 1], o[r], o[4 + r], most[r]);
                        }
                    };
                    uint32_t held[kGrp][8];
                    const bool two = Np > kPh;
                    if (two) {
                        if (!wait_acc(kPh)) { ok = false; break; }
                        groups(share, kPh, kPh, kPh, act, act, [&](int i, int, const uint32_t (&o)[8]) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) held[i][k] = o[k];
                        });
                        drained();
                    }
                    const int n0 = two ? kPh : 0;
                    if (!wait_acc(Np - n0)) { ok = false; break; }
                    if (two && !last) {
#pragma unroll
                        for (int i = 0; i < kGrp; ++i)
                            if (pt + i * kParts < kPh / 8) store4(rh, rl, 8 * (pt + i * kParts), held[i]);
                        operand_done(0);
                    }
                    auto rest = [&](int c, const float (&z)[8], uint32_t (&o)[8]) { act(n0 + c, z, o); };
                    groups(share, Np - n0, Np - n0, Np - n0, rest, rest, [&](int, int c, const uint32_t (&o)[8]) {
                        if (!last) store4(rh, rl, n0 + c, o);
                    });
                    drained();
                    if (!last) {
                        operand_done(two ? 1 : 0);
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const int at = kTile * r + 8 * q + sq;
                            if (reaches(most[r])) s_act[(L - LS) * 128 + at] = 1;
                            if (out_of_range(most[r])) s_bad[at] = 1;
                        }
                        continue;
                    }
                    // ---- the next unit's first layer-0 input (every MMA of this one is complete), the colours ----
#pragma unroll
                    for (int k = 0; k < 3; ++k)
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            cd[k][r] += __shfl_xor_sync(0xffffffffu, cd[k][r], 1);
                            cd[k][r] += __shfl_xor_sync(0xffffffffu, cd[k][r], 2);
                            if ((lane & 3) == 0) s_cdot[(pt * 3 + k) * 128 + 32 * q + 8 * r + sq] = cd[k][r] * (1.0f / kUp);
                        }
                    if (!epi_sync()) { ok = false; break; }
                    if (kt + 1 < mine) write_input0();
                    if (et < 128) {
                        const float* bc = p.rgb_w + F::param_offset(F::NL - 1) + 3 * F::layer(F::NL - 1).in;
                        const int j = (et >> 3) & 3, s = 8 * (et >> 5) + (et & 7);   // tile of the unit, its sample
                        const int64_t g = tile_of(kt - slot + j) * kTile + s;
                        bool bad = s_bad[kTile * j + s] != 0;
                        s_bad[kTile * j + s] = 0;
                        for (int l = 0; l < F::kChecked; ++l) {
                            bad = bad || s_act[l * 128 + kTile * j + s] == 0;
                            s_act[l * 128 + kTile * j + s] = 0;
                        }
                        if (j <= slot && g < total) {
                            float* R = reinterpret_cast<float*>(p.rec + g);
#pragma unroll
                            for (int k = 0; k < 3; ++k) {
                                const float* sd = s_cdot + k * 128 + et;
                                const float c3 = sd[0] + sd[3 * 128] + sd[6 * 128] + __ldg(bc + k);
                                bad = bad || !(fabsf(c3) < __int_as_float(0x7f800000));
                                R[4 + k] = 1.0f / (1.0f + expf(-c3));
                            }
                            if (bad || *s_low != 0) {
                                p.rec[g].pad = 1.0f;
                                atomicExch(p.redo, 1u);
                            }
                        }
                    }
                }
            }
        }
        if (!ok) set_status(p.status, TSDFS_DEV_TIMEOUT);
        if (!ok && backs > 0) {   // this thread's copies may be in flight
            for (uint32_t it = 0; it < kMaxSpin && !mbar_try(bar_back, (backs - 1) & 1u); ++it) {
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kMma) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

// Split the parameters into the items' hi and lo images (8 x 8 core matrices, K-major), one
// 8-column row piece per thread; clears the redo words, and tells for each layer whether all its weights
// are below kFloor (a block per layer, which looks at 256 of them with ordinary weights).  3 MB for the
// room networks, every call: the parameters may have changed since the last one.
template <int ARCH>
__global__ void k_split_weights(const float* __restrict__ sdf_w, const float* __restrict__ rgb_w,
                                uint8_t* __restrict__ packed, uint32_t* __restrict__ redo) {
    using F = FArch<ARCH>;
    if (blockIdx.x == 0 && threadIdx.x == 0) redo[0] = redo[1] = 0;
    for (int L = blockIdx.x; L < F::NL - 1; L += gridDim.x) {
        const Layer ly = F::layer(L);
        const float* W = (L < F::LS ? sdf_w : rgb_w) + F::param_offset(L);
        const int n = ly.out * ly.in;
        int i = L == F::LS - 1 ? ly.in : 0;   // the SDF output's features: net_0's row is no operand
        bool fine = false, some = false;      // a weight that reaches kFloor, one that is not 0
        for (; i < n && !fine; i += blockDim.x) {
            const float w = i + (int)threadIdx.x < n ? fabsf(__ldg(W + i + threadIdx.x)) : 0.0f;
            some = some || w != 0.0f;
            fine = __syncthreads_or(!(w < kFloor)) != 0;
        }
        if (!fine) some = __syncthreads_or(some) != 0;
        if (threadIdx.x == 0) redo[kLowWord + L] = !fine && some ? 1u : 0u;
    }
    constexpr int64_t n8 = F::packed_bytes() / 32;   // 8 columns x 2 parts x 2 bytes
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n8; i += (int64_t)gridDim.x * blockDim.x) {
        int L = 0;
        while (L + 2 < F::NL && F::layer_base(L + 1) <= i * 32) ++L;
        const Layer ly = F::layer(L);
        int64_t r = i - F::layer_base(L) / 32;     // within the layer, in items' order
        const int kt = (F::k_main(L) + (L == F::LS ? F::kXp : 0)) / 8;
        int ph = 0, n_first = 0;
        while (r >= (int64_t)F::phase_n(L, ph) * kt) {
            r -= (int64_t)F::phase_n(L, ph) * kt;
            n_first += F::phase_n(L, ph++);
        }
        const int n_ph = F::phase_n(L, ph);
        int c = 0, k_first = 0;
        while (r >= (int64_t)n_ph * (F::chunk_k(L, c) / 8)) {
            r -= (int64_t)n_ph * (F::chunk_k(L, c) / 8);
            k_first += F::chunk_k(L, c++);
        }
        const int kc8 = F::chunk_k(L, c) / 8;
        const int n = (int)(r / kc8), k8 = (int)(r % kc8);
        const int row = F::src_row(L, n_first + n);
        const float* W = (L < F::LS ? sdf_w : rgb_w) + F::param_offset(L);
        uint32_t o[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float v[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int col = F::src_col(L, k_first + 8 * k8 + 2 * j + e);
                v[e] = row >= 0 && col >= 0 ? __ldg(W + (int64_t)row * ly.in + col) : 0.0f;
            }
            split_f32(v[0] * kUp, v[1] * kUp, o[j], o[4 + j]);
        }
        // the item's hi image starts after the phases and chunks before it
        uint8_t* item = packed + F::layer_base(L) + (int64_t)n_first * kt * 32 + (int64_t)n_ph * (k_first / 8) * 32;
        const uint32_t at = (uint32_t)(((n >> 3) * kc8 + k8) * 128 + (n & 7) * 16);
        *reinterpret_cast<uint4*>(item + at) = make_uint4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<uint4*>(item + (int64_t)n_ph * kc8 * 16 + at) = make_uint4(o[4], o[5], o[6], o[7]);
    }
}

template <int ARCH, bool VALUE>
int launch_f32(const tsdfs_mlp* m, const SampleSource& src, SampleRec* rec, float* f_out, int64_t max_samples,
               Scratch stash, cudaStream_t st) {
    using F = FArch<ARCH>;
    constexpr size_t smem = F::template smem_bytes<VALUE>();
    static_assert(smem <= 232448, "k_mlp_f32 shared memory exceeds 227 KB");
    static std::mutex mu;
    static bool set[64] = {};
    int dev = 0, sms = 152;
    int rc = cuda_check(cudaGetDevice(&dev), "mlp_f32 device");
    if (rc) return rc;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (dev < 0 || dev >= 64 || !set[dev]) {
            rc = cuda_check(cudaFuncSetAttribute(k_mlp_f32<ARCH, VALUE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem),
                            "mlp_f32 smem attribute");
            if (rc) return rc;
            if (dev >= 0 && dev < 64) set[dev] = true;
        }
    }
    F32Params p{};
    constexpr size_t head = kRedoBytes + F::packed_bytes();
    p.packed = stash.at + kRedoBytes;
    p.park = stash.at + head;
    p.redo = reinterpret_cast<uint32_t*>(stash.at);
    p.sdf_w = m->sdf_w;
    p.rgb_w = m->rgb_w;
    for (int a = 0; a < 3; ++a) p.center[a] = m->center[a];
    p.scale = m->scale;
    p.inv_scale = 1.0f / m->scale;
    p.beta = m->beta;
    p.src = src;
    p.rec = rec;
    p.f_out = f_out;
    p.status = device_status_word();
    p.spin = test_spin_limit(kMaxSpin);
    p.withhold = test_withhold_chunk();
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t ts = VALUE ? kTileV : kTile, tiles = (max_samples + ts - 1) / ts;
    const int64_t places = (int64_t)((stash.bytes - head) / F::park_bytes());
    if (!VALUE && sms > places) sms = (int)places;
    const unsigned blocks = (unsigned)(tiles < sms ? (tiles < 1 ? 1 : tiles) : sms);
    k_split_weights<ARCH><<<grid_1d(F::packed_bytes() / 32, 256), 256, 0, st>>>(m->sdf_w, m->rgb_w,
                                                                               stash.at + kRedoBytes, p.redo);
    k_mlp_f32<ARCH, VALUE><<<blocks, kThr, smem, st>>>(p);
    return cuda_check(cudaGetLastError(), "mlp_f32 launch");
}

}  // namespace

size_t mlp_f32_stash_bytes(int arch) {
    auto bytes = [](auto f) {
        using F = decltype(f);
        return kRedoBytes + (size_t)F::packed_bytes() + kMaxCtas * F::park_bytes();
    };
    return arch == TSDFS_ARCH_TINY ? bytes(FArch<TSDFS_ARCH_TINY>{}) : bytes(FArch<TSDFS_ARCH_ROOM>{});
}

int launch_mlp_full_f32(const tsdfs_mlp* m, const SampleSource& src, SampleRec* rec, int64_t max_samples,
                        Scratch stash, cudaStream_t st) {
    return m->arch == TSDFS_ARCH_TINY ? launch_f32<TSDFS_ARCH_TINY, false>(m, src, rec, nullptr, max_samples, stash, st)
                                      : launch_f32<TSDFS_ARCH_ROOM, false>(m, src, rec, nullptr, max_samples, stash, st);
}

int launch_mlp_value_f32(const tsdfs_mlp* m, const SampleSource& src, float* f_out, Scratch stash, cudaStream_t st) {
    const int64_t n = sample_bound(src);
    return m->arch == TSDFS_ARCH_TINY ? launch_f32<TSDFS_ARCH_TINY, true>(m, src, nullptr, f_out, n, stash, st)
                                      : launch_f32<TSDFS_ARCH_ROOM, true>(m, src, nullptr, f_out, n, stash, st);
}

}  // namespace tsdfs
