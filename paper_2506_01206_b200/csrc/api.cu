// C ABI of the library: argument checks, launch planning, dispatch.  Nothing here allocates or keeps state between
// calls (the one exception in the library is the fixed scratch array of mdraft_conv_scan_prefill_noalloc, noalloc.cu).
#include <cudaTypedefs.h>
#include <limits.h>

#include <string.h>

#include <atomic>

#include "block.cuh"
#include "commit.cuh"
#include "common.cuh"
#include "prefill.cuh"
#include "prefill_cluster.cuh"
#include "ssd.cuh"
#include "tree_proj.cuh"
#include "tree_step.cuh"

using namespace mdraft;

// SMs of the current device; the B200's count when no device can be asked (the workspace query also runs where there
// is none, and must then give the size the call will want on the B200 it is planned for).
int mdraft::sm_count() {
    constexpr int kSmCountB200 = 148;
    static std::atomic<int> known{0};  // every device this library runs on is the same part
    int dev = 0, n = known.load(std::memory_order_relaxed);
    if (n > 0) return n;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
        (void)cudaGetLastError();
        return kSmCountB200;
    }
    known.store(n, std::memory_order_relaxed);
    return n;
}

namespace {

inline size_t elem_size(int act) { return act == MDRAFT_BF16 ? 2 : 4; }
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

int check_layer(const mdraft_layer* L) {
    if (!L || !L->A || !L->conv_w) return MDRAFT_ERR_INVALID_ARG;
    if (L->d_inner <= 0) return MDRAFT_ERR_INVALID_ARG;
    if (L->d_state != kN || L->d_conv != kW || (L->d_inner % 8) != 0) return MDRAFT_ERR_UNSUPPORTED;
    if (L->act != MDRAFT_F32 && L->act != MDRAFT_BF16) return MDRAFT_ERR_UNSUPPORTED;
    if ((L->flags & MDRAFT_PRECONV) && (L->flags & MDRAFT_CONV_ONLY)) return MDRAFT_ERR_INVALID_ARG;
    if (!aligned16(L->A) || !aligned16(L->conv_w)) return MDRAFT_ERR_MISALIGNED;
    return MDRAFT_OK;
}

int check_cache(const mdraft_cache* c, int d_inner, int act, int layer_index, int d_state = kN) {
    if (!c || !c->ssm || !c->conv) return MDRAFT_ERR_INVALID_ARG;
    if (c->n_layers <= 0 || c->n_slots <= 0 || layer_index < 0 || layer_index >= c->n_layers) return MDRAFT_ERR_INVALID_ARG;
    const int64_t ssm_elems = (int64_t)d_inner * d_state, conv_elems = (int64_t)(kW - 1) * d_inner;
    if (c->ssm_slot_stride < ssm_elems || c->conv_slot_stride < conv_elems) return MDRAFT_ERR_INVALID_ARG;
    if (c->n_layers > 1 && (c->ssm_layer_stride < 0 || c->conv_layer_stride < 0)) return MDRAFT_ERR_INVALID_ARG;
    const size_t es = elem_size(act);
    if (!aligned16(c->ssm) || !aligned16(c->conv)) return MDRAFT_ERR_MISALIGNED;
    if ((c->ssm_slot_stride * 4) % 16 || (c->ssm_layer_stride * 4) % 16 || (c->conv_slot_stride * es) % 16 ||
        (c->conv_layer_stride * es) % 16)
        return MDRAFT_ERR_MISALIGNED;
    return MDRAFT_OK;
}

int check_matrix(const void* p, int64_t ld, int cols, int act, bool required) {
    if (!p) return required ? MDRAFT_ERR_INVALID_ARG : MDRAFT_OK;
    if (ld < cols) return MDRAFT_ERR_INVALID_ARG;
    if (!aligned16(p) || (ld * (int64_t)elem_size(act)) % 16) return MDRAFT_ERR_MISALIGNED;
    return MDRAFT_OK;
}

// Flags beyond softplus and A = powers: the split modes and raw step sizes, which have kernels of their own that take one layer.
bool one_at_a_time(const mdraft_layer* layer) { return (layer->flags & ~(uint32_t)MDRAFT_A_POWERS) != (uint32_t)MDRAFT_DT_SOFTPLUS; }

LayerDev layer_dev(const mdraft_layer* L) {
    LayerDev d;
    d.A = L->A; d.D = L->D; d.conv_w = L->conv_w; d.conv_b = L->conv_b; d.dt_bias = L->dt_bias;
    d.d_inner = L->d_inner; d.flags = L->flags;
    return d;
}

PoolDev pool_dev(const mdraft_cache* c, int act, int layer_index) {
    PoolDev p;
    p.ssm = c->ssm + (int64_t)layer_index * c->ssm_layer_stride;
    p.conv = static_cast<char*>(c->conv) + (int64_t)layer_index * c->conv_layer_stride * (int64_t)elem_size(act);
    p.ssm_slot_stride = c->ssm_slot_stride;
    p.conv_slot_stride = c->conv_slot_stride;
    p.n_slots = c->n_slots;
    return p;
}

struct PrefillPlan {
    int chunk_len;       // tokens per chunk (INT_MAX/2 when every sequence is one chunk)
    int n_chunks_bound;  // upper bound on the number of chunks
    PrefillForm form;
    bool longest_first;  // unsplit sequences of different lengths, handed out longest first
    size_t off_q, off_sd, off_h0, off_conv, layer_bytes;
    size_t bytes;        // what the workspace query answers: the call's layers, split
};

// Chunk length: split the token axis until every SM holds three blocks of kPrefillThreads channels, or one wide block
// (one resident wave, no tail).  Narrow blocks have more registers a thread, hide one another's set-up and can be 16 tokens
// short; wide ones take fewer cycles a token.  Measured (one layer, narrow against wide): 1536 channels x 256 tokens 15.0
// against 26.0 us, 512 x 4096 27.5 against 31.0, 1536 x 2048 34.4 against 32.7 with A = powers and 41.7 against 42.5 with a
// general A, 1536 x 32768 357 against 338 and 507 against 491: narrow while one wave of them takes chunks of at most
// kNarrowChunk (kNarrowChunkGeneral) tokens.
// Where one sequence is one or two channel blocks wide, chunks of less than a 128th of it (to the nearest 8 tokens, beyond 40 to the next) cost the carry scan
// more than they give the passes (3000 tokens x 64 / 128 / 192 channels: 16-token chunks 16.8 / 18.3 / 20.4 us, 24-token 15.7 / 16.8 /
// 18.8; 4000 x 64 / 256: 16-token 20.1 / 25.4, 32-token 16.7 / 24.9), up to kOneBlockChunk tokens for one channel block, whose chunks then
// have an SM each (5000 x 128: 32-token 23.1, 40-token 20.4; 6976 x 112, general A: 31.7, 56-token 28.1; 8000 x 64: 23.9, 64-token
// 24.9, two blocks of 32 tokens an SM again), and up to kMinChunkWide for two; with more channel blocks, or with two and a general A, whose passes
// cost more, they pay (3300 x 256, general A: 16-token chunks 23.3, 24 25.5, 32 28.3; 3000 x 384: 21 23.1, 32 23.5).
// When one wave of narrow blocks would need longer chunks, a single sequence takes one wave of wide blocks, or, where its width
// does not fill them, several waves of kManyWavesChunk tokens once one wave would need more than kOneWaveMax.  Packed batches,
// whose chunks are uneven, take one to three waves of narrow blocks, kManyWavesMin to kManyWavesChunk tokens a chunk: blocks are
// handed out as SMs free up, which evens them out (8 x 2000 tokens x 512 channels: wide 83.7 us, 48-64 tokens 73.5, 128 79.8; 26
// sequences of 4k-12k tokens x 152 channels: 64 tokens 331, 128 321, 256 334).
// Three narrow blocks to an SM have 128 registers a thread, four have 96.  Four are up to 17 % faster where the width leaves a warp of each
// block idle and the batch is packed (32 sequences, 91k tokens x 72 channels 94.7 -> 85.1 us; 20, 37k x 88, general A 59.3 -> 48.8;
// 32, 17k x 288 72.2 -> 65.6), slower elsewhere (full blocks, general A: 2-5 %; one sequence of 13608 x 96 38.7 -> 41.6).
constexpr int kMinChunk = 16, kMinChunkWide = 32, kNarrowChunk = 48, kNarrowChunkGeneral = 72;
constexpr int kOneWaveMax = 256, kManyWavesChunk = 128, kManyWavesMin = 48, kOneWaveNarrow = 110, kOneBlockChunk = 56;

// Splitting a sequence costs a second pass over its tokens (0.75 of the output pass, for all chunks but the last) and two more
// launches; not splitting it leaves one block per sequence, layer and 128 or 256 channels.  SM cycles a token of a block takes
// (A = powers), measured: a block of 128 channels alone on its SM, one of 256 channels alone,
// three of 128 side by side (per block; in many waves of short chunks, and in one wave of unsplit sequences), and a wide one per
// 128 channels.  Blocks that share an SM are not served evenly (of two,
// one ran 548k cycles and the other 708k over the same 2048 tokens) and the last one finishes alone at the rate of one warp per
// scheduler; the warps of one block advance together.  Hence 256 channels in one block rather than two blocks of 128.
constexpr double kCycOne = 205, kCycPair = 315, kCycMany = 170, kCycCrowd = 204, kCycWide = 146, kSplitCycles = 20500, kOffsetCycles = 5000, kBlockCycles = 6500;
constexpr double kGeneralOne = 1.38, kGeneralMany = 1.26;   // a general A takes so much more: few warps per scheduler, many
constexpr double kFloatOne = 1.1;                            // fp32 activations, few warps per scheduler

// Estimated cycles of the unsplit form with one block per SM: the longest sequence, or what the fullest SM is given.
double unsplit_cycles(int64_t blocks_per_seq, double cycles, int T, int n_seq, int max_seqlen, int sms) {
    const int64_t rounds = (blocks_per_seq * n_seq + sms - 1) / sms;
    double m = (double)blocks_per_seq * T / sms + 0.5 * T / n_seq;   // longest first: the last blocks to start are the short ones
    if (m > (double)rounds * max_seqlen) m = (double)rounds * max_seqlen;
    if (m < max_seqlen) m = max_seqlen;
    return cycles * m + kBlockCycles * rounds;
}

// Workspace of one layer with this many chunks; with `pl`, where its parts lie.
size_t workspace_of(const mdraft_layer* L, int n_seq, int chunks, PrefillPlan* pl = nullptr) {
    const size_t Dz = (size_t)L->d_inner;
    const size_t sd = align_up((size_t)chunks * Dz * kN * sizeof(float), 256);
    const size_t h0 = align_up(sd + (size_t)chunks * Dz * sizeof(float), 256);
    const size_t conv = align_up(h0 + (size_t)n_seq * Dz * kN * sizeof(float), 256);
    if (pl) { pl->off_q = 0; pl->off_sd = sd; pl->off_h0 = h0; pl->off_conv = conv; }
    return align_up(conv + (size_t)n_seq * (kW - 1) * Dz * elem_size(L->act), 256);
}

constexpr size_t kAnyWorkspace = SIZE_MAX;  // "whatever the plan asks for"

// workspace: bytes that the call has.  A call that has fewer than the plan would like gets fewer chunks; one that has fewer than
// the longest chunks need gets a plan with bytes > workspace, which the caller refuses.
PrefillPlan plan_prefill(const mdraft_layer* L, int n_layers, int T, int n_seq, int max_seqlen, const mdraft_prefill_opts* opts, size_t workspace) {
    PrefillPlan pl;
    const int D = L->d_inner;
    const int wide_cols = kPrefillThreads * kPrefillWideBoxes;
    const int64_t ch_blocks = (int64_t)n_layers * ((D + kPrefillThreads - 1) / kPrefillThreads);
    const int64_t ch_blocks_wide = (int64_t)n_layers * ((D + wide_cols - 1) / wide_cols);
    const int64_t ch_blocks_pair = (int64_t)n_layers * ((D + 2 * kPrefillThreads - 1) / (2 * kPrefillThreads));
    const int forced = opts ? opts->block_channels : 0;
    const int sms = sm_count();
    // Wide blocks pay off when they fill the machine in one wave: every SM then runs ONE block whose 16 channel warps
    // advance together and finish together (narrow blocks side by side finish one after another and leave the SM to
    // the last of them).  They need the channel count to (nearly) fill whole 512-channel blocks.
    bool wide = forced == wide_cols || (forced == 0 && ch_blocks_wide * wide_cols * 9 <= (int64_t)n_layers * D * 10);
    int Lc;
    bool unsplit = false, alone = false, four = false;
    int unsplit_boxes = 1;
    const bool general = !(L->flags & MDRAFT_A_POWERS);
    if (opts && opts->chunk_len > 0) {
        Lc = opts->chunk_len < 4 ? 4 : opts->chunk_len;
    } else {
        // Four narrow blocks to an SM instead of three: for packed batches whose blocks have a warp of four to spare (the width fills at
        // most three quarters of them) and whose wave of four takes whole tiles; with several channel blocks for A = powers only.
        four = n_layers == 1 && n_seq > 1 && !one_at_a_time(L) && (D + 31) / 32 <= 3 * ch_blocks && (!general || ch_blocks == 1) &&
               T >= kMinChunk * (sms * 4 / ch_blocks - (n_seq - 1) / 2);
        const int per_sm = four ? 4 : 3;
        // Chunks of a wave of so many blocks to an SM; every sequence leaves its last chunk half unfilled, on average.
        auto wave_chunks = [&](int blocks) { return sms * blocks / ch_blocks - (n_seq - 1) / 2; };
        auto wave_length = [&](int blocks) { return wave_chunks(blocks) > 0 ? (T + wave_chunks(blocks) - 1) / wave_chunks(blocks) : (int64_t)(INT_MAX / 2); };
        const int64_t want_narrow = wave_chunks(per_sm), even = wave_length(per_sm);
        int shortest = max_seqlen / 128;
        if (n_seq == 1) shortest = ch_blocks == 1 || (ch_blocks == 2 && !general) ? (shortest + (shortest > 40 ? 7 : 4)) / 8 * 8 : kMinChunk;
        const int most_shortest = n_seq == 1 && ch_blocks == 1 && shortest <= kOneBlockChunk ? kOneBlockChunk : kMinChunkWide;
        shortest = shortest < kMinChunk ? kMinChunk : shortest > most_shortest ? most_shortest : shortest;
        const int64_t narrow = even < shortest ? shortest : even;
        const bool short_chunks = narrow * per_sm <= (general ? kNarrowChunkGeneral : kNarrowChunk) * 3;
        // The longest chunks that a call is given when its workspace does not hold the preferred ones: one wide block or four narrow ones to
        // an SM, at least kMinChunkWide tokens and, for several sequences, at most kOneWaveMax (`coarse`); three narrow ones where that
        // is what a wave of short chunks may be.  Where not even those fit, leaving the sequences whole is weighed against `coarse` chunks.
        const int64_t most = wide ? sms / ch_blocks_wide : sms * 4 / ch_blocks, uncapped = (T + (most < 1 ? 1 : most) - 1) / (most < 1 ? 1 : most);
        const bool coarse_wide = wide && (n_seq == 1 || uncapped <= kOneWaveMax);
        const int64_t coarse = uncapped < kMinChunkWide ? kMinChunkWide : uncapped > kOneWaveMax && n_seq > 1 ? kOneWaveMax : uncapped;
        if (forced == 0 && short_chunks) wide = false;
        int64_t longest = !wide && (n_seq == 1 || four) ? wave_length(3) : coarse;
        if (n_seq > 1 && longest > kOneWaveMax) longest = kOneWaveMax;
        if (longest < coarse) longest = coarse;
        if (wide) {
            int64_t want = sms / ch_blocks_wide;
            if (want < 1) want = 1;
            Lc = (int)((T + want - 1) / want);
            if (Lc < kMinChunkWide) Lc = kMinChunkWide;
        } else {
            Lc = (int)narrow;
            // One sequence: where whole tiles would leave a few tokens over a full wave, those make a short last chunk instead of one more
            // step for every chunk.  It starts when the wave's first blocks are done and is hidden while it is shorter than they finish
            // apart: up to a third of a chunk and 16 tokens (1536 channels, general A, 48-token chunks against 49: 1777 tokens 37.8
            // and 39.2 us, 1790 38.5 and 39.1; against 50: 1821 42.6 and 39.9.  16 against 17: 596 17.3 and 17.0, 601 17.7 and 17.0).
            const int tile = kPrefillTileRowBytes / (int)elem_size(L->act), down = (int)narrow / tile * tile;
            const int64_t over = T - want_narrow * down;
            if (n_seq == 1 && narrow == even && down >= kMinChunk && over <= 16 && over * 3 <= down) Lc = down;
        }
        // A single sequence in wide blocks stays in one wave at any length: 49 x 3 equal chunks finish together
        // (32768 tokens: 344 us against 372-376 for several waves of short chunks; 65536: 675 against 724).
        if (n_seq == 1) {
            if (Lc > kOneWaveMax && !wide) Lc = kManyWavesChunk;
        } else if (forced == 0 && !short_chunks) {
            // One wave while its chunks are short and the sequences' unfilled last chunks few (5 x 3172 tokens x 256 channels: 73-token
            // chunks 53.9 us, 48 59.6), then two, then three.
            const int64_t one_wave = narrow * per_sm / 3;   // tokens a chunk of a wave of three blocks to an SM
            int64_t waves = one_wave <= kOneWaveNarrow && n_seq * narrow * 20 <= T ? narrow : narrow / (one_wave <= 2 * kOneWaveNarrow ? 2 : 3);
            waves = waves < kManyWavesMin ? kManyWavesMin : waves > kManyWavesChunk ? kManyWavesChunk : waves;
            Lc = (int)waves;
            wide = false;
        } else if (Lc > kOneWaveMax) {
            Lc = kOneWaveMax;
            if (forced == 0) wide = false;
        }
        if (n_seq + (int64_t)T / Lc > 65535 && Lc < kOneWaveMax) Lc = kOneWaveMax;  // a launch's grid
        const double g1 = (general ? kGeneralOne : 1.0) * (L->act == MDRAFT_F32 ? kFloatOne : 1.0), gm = general ? kGeneralMany : 1.0;
        // The unsplit forms: 128 channels alone, 256 channels alone, and three blocks of 128 channels to an SM for many short sequences.
        const double one = unsplit_cycles(ch_blocks, g1 * kCycOne, T, n_seq, max_seqlen, sms), pair = unsplit_cycles(ch_blocks_pair, g1 * kCycPair, T, n_seq, max_seqlen, sms);
        double many = gm * kCycCrowd * ((double)ch_blocks * T / sms + 0.7 * max_seqlen);   // uneven neighbours on an SM
        if (many < g1 * kCycOne * max_seqlen) many = g1 * kCycOne * max_seqlen;
        many += kBlockCycles;
        auto better_whole = [&](int64_t chunk, bool wide_blocks) {
            const double n_chunks = n_seq + (double)T / chunk, work = (double)ch_blocks * T / sms * (wide_blocks ? kCycWide * g1 : kCycMany * gm);
            const double split = (work > g1 * kCycOne * chunk ? work : g1 * kCycOne * chunk) * (1.0 + 0.75 * (n_chunks - n_seq) / n_chunks) + kSplitCycles + (n_seq > 1 ? kOffsetCycles : 0.0);
            return forced == 0 && (one <= split || pair <= split || many <= split);
        };
        unsplit = better_whole(Lc, wide);
        auto need = [&](int64_t len) { return len < max_seqlen ? n_layers * workspace_of(L, n_seq, (int)(n_seq + T / len)) : (size_t)0; };
        if (!unsplit && need(Lc) > workspace) {
            if (Lc < longest) {  // the shortest chunks that fit, in whole groups of tokens
                int64_t lo = Lc, hi = longest;  // need(lo) > workspace; need() falls with the length
                while (hi - lo > 1) (need((lo + hi) / 2) > workspace ? lo : hi) = (lo + hi) / 2;
                hi = (hi + 7) / 8 * 8;
                Lc = (int)(hi < longest ? hi : longest);
            }
            unsplit = need(Lc) > workspace ? better_whole(coarse, coarse_wide) : better_whole(Lc, wide);
        }
        if (unsplit) {
            unsplit_boxes = pair < one && pair < many ? 2 : 1;
            alone = unsplit_boxes == 2 || one <= many;
        }
    }
    pl.form.boxes = unsplit ? unsplit_boxes : wide ? kPrefillWideBoxes : 1;
    pl.form.chunked = Lc < max_seqlen;
    pl.longest_first = pl.form.alone = false;
    pl.form.four = four && !unsplit && !wide;
    pl.chunk_len = INT_MAX / 2;
    pl.n_chunks_bound = n_seq;
    pl.off_q = pl.off_sd = pl.off_h0 = pl.off_conv = pl.layer_bytes = pl.bytes = 0;
    if (pl.form.chunked) {
        const int bound = n_seq + T / Lc;
        pl.layer_bytes = workspace_of(L, n_seq, bound, &pl);
        // For one layer the query answers for the split form whichever form is taken: a workspace made for one batch then
        // serves another of its size whose longest sequence is longer.
        pl.bytes = pl.layer_bytes * n_layers;
        if (!unsplit) {
            pl.chunk_len = Lc;
            pl.n_chunks_bound = bound;
        }
    }
    if (unsplit) {
        pl.form.chunked = false;
        // Where every block starts at once the order is worth nothing.
        const bool at_once = (pl.form.boxes == 2 ? ch_blocks_pair : ch_blocks) * n_seq <= sms;
        pl.longest_first = !at_once && n_seq > 1 && n_seq <= kPrefillMaxRanked;
        pl.form.alone = alone;
    }
    return pl;
}

// cuTensorMapEncodeTiled, fetched through the runtime so that the library has no link-time dependency on the
// driver (it can then be loaded, and its host-side checks exercised, on a machine without one).
PFN_cuTensorMapEncodeTiled tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) f = nullptr;
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled>(f);
    }();
    return fn;
}

// Descriptor of a (rows x cols) row-major activation matrix with row stride ld, read in boxes of box_cols x tile rows.
bool encode_matrix(CUtensorMap* m, const void* base, int act, int64_t rows, int64_t cols, int64_t ld, int box_cols) {
    PFN_cuTensorMapEncodeTiled enc = tensor_map_encoder();
    if (!enc) return false;
    if (!base) {  // tensor not used by this mode: leave a recognisable empty descriptor
        memset(m, 0, sizeof(*m));
        return true;
    }
    const cuuint64_t es = elem_size(act);
    cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t gstride[1] = {(cuuint64_t)ld * es};
    cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)(kPrefillTileRowBytes / es)};
    cuuint32_t estride[2] = {1, 1};
    return enc(m, act == MDRAFT_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base),
               gdim, gstride, box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Arguments of a call over several layers: the layers share a cache, so width, states, taps and type must agree.
int check_stack(int32_t n_layers, const mdraft_layer* layers, const int32_t* layer_index, const mdraft_io* io) {
    if (n_layers <= 0 || !layers || !layer_index || !io) return MDRAFT_ERR_INVALID_ARG;
    for (int32_t i = 0; i < n_layers; ++i) {
        if (int rc = check_layer(layers + i)) return rc;
        if (layers[i].d_inner != layers->d_inner || layers[i].act != layers->act) return MDRAFT_ERR_UNSUPPORTED;
    }
    return MDRAFT_OK;
}

int check_io(const mdraft_io& v, const mdraft_layer& L, bool required) {
    const bool all = required && !(L.flags & MDRAFT_CONV_ONLY);
    int rc;
    if ((rc = check_matrix(v.x, v.ldx, L.d_inner, L.act, required))) return rc;
    if ((rc = check_matrix(v.out, v.ldo, L.d_inner, L.act, required))) return rc;
    if ((rc = check_matrix(v.z, v.ldz, L.d_inner, L.act, all))) return rc;
    if ((rc = check_matrix(v.dt, v.lddt, L.d_inner, L.act, all))) return rc;
    if ((rc = check_matrix(v.B, v.ldb, kN, L.act, all))) return rc;
    return check_matrix(v.C, v.ldc, kN, L.act, all);
}

// How many of the next n layers one launch takes: those with the first one's flags, at most `most`.
int32_t run_length(int32_t n, const mdraft_layer* layers, int32_t most) {
    if (one_at_a_time(layers)) return 1;
    int32_t k = 1;
    while (k < n && k < most && layers[k].flags == layers->flags) ++k;
    return k;
}

// Layers that one launch of the prefill may take: its grid's last dimension also counts sequences (in the carry scan).
int32_t prefill_most_layers(int32_t n_seq) { return n_seq > 65535 / kPrefillMaxLayers ? 1 : kPrefillMaxLayers; }

// The launches of a prefill of n_layers layers with this one's flags: f(layers of a launch, how many such launches).
template <typename F>
void for_each_prefill_run(const mdraft_layer* layer, int32_t n_layers, int32_t n_seq, F&& f) {
    const int32_t most = one_at_a_time(layer) ? 1 : prefill_most_layers(n_seq);
    if (n_layers >= most) f(most, n_layers / most);
    if (n_layers % most) f(n_layers % most, 1);
}

struct PrefillCall {
    const mdraft_cache* cache;
    int32_t total_tokens, n_seq;
    const int32_t *cu_seqlens, *init_slot, *final_slot;
    char* workspace;
    const mdraft_prefill_opts* opts;
    int32_t* dev_status;
    cudaStream_t stream;
};

// One launch sequence of the prefill over n_layers (at most ML) layers with the same flags.
template <int ML>
int run_prefill(const PrefillCall& call, const PrefillPlan& pl, int32_t n_layers, const mdraft_layer* layers, const int32_t* layer_index, const mdraft_io* io) {
    PrefillBatch<ML> b;
    PrefillArgs& a = b.c;
    const int act = layers->act, D = layers->d_inner;
    if (call.cache) {
        a.pool = pool_dev(call.cache, act, 0);
        a.ssm_layer_stride = call.cache->ssm_layer_stride; a.conv_layer_stride = call.cache->conv_layer_stride;
    } else {
        a.pool.ssm = nullptr; a.pool.conv = nullptr; a.pool.ssm_slot_stride = 0; a.pool.conv_slot_stride = 0; a.pool.n_slots = 0;
        a.ssm_layer_stride = a.conv_layer_stride = 0;
    }
    a.n_layers = n_layers; a.d_inner = D;
    a.T = call.total_tokens; a.n_seq = call.n_seq; a.chunk_len = pl.chunk_len; a.n_chunks_bound = pl.n_chunks_bound;
    a.longest_first = pl.longest_first;
    a.cu = call.cu_seqlens; a.init_slot = call.init_slot; a.final_slot = call.final_slot;
    char* ws = call.workspace;
    a.ws_q = pl.form.chunked ? reinterpret_cast<float*>(ws + pl.off_q) : nullptr;
    a.ws_sd = pl.form.chunked ? reinterpret_cast<float*>(ws + pl.off_sd) : nullptr;
    a.ws_h0 = pl.form.chunked ? reinterpret_cast<float*>(ws + pl.off_h0) : nullptr;
    a.ws_conv = pl.form.chunked ? static_cast<void*>(ws + pl.off_conv) : nullptr;
    a.ws_layer_bytes = (int64_t)pl.layer_bytes;
    a.dev_status = call.dev_status;
    a.pdl_inputs_ready = pl.form.chunked ? 1 : 0;  // the summary pass waits for the producer of the inputs on behalf of all three kernels
    a.ev_state = call.opts ? static_cast<cudaEvent_t>(call.opts->event_after_chunk_state) : nullptr;
    a.ev_carry = call.opts ? static_cast<cudaEvent_t>(call.opts->event_after_carry_scan) : nullptr;
    const bool rows = call.total_tokens > 0;  // with no tokens at all (only empty sequences) nothing is ever copied: empty descriptors
    for (int32_t i = 0; i < n_layers; ++i) {
        PrefillLayer& p = b.l[i];
        const mdraft_io& v = io[i];
        p.L = layer_dev(layers + i);
        p.layer_index = layer_index[i];
        p.x = v.x; p.ldx = v.ldx; p.out = v.out; p.ldo = v.ldo;
        if (!encode_matrix(&p.maps.x, rows ? v.x : nullptr, act, a.T, D, v.ldx, kPrefillThreads) ||
            !encode_matrix(&p.maps.dt, rows ? v.dt : nullptr, act, a.T, D, v.lddt, kPrefillThreads) ||
            !encode_matrix(&p.maps.z, rows ? v.z : nullptr, act, a.T, D, v.ldz, kPrefillThreads) ||
            !encode_matrix(&p.maps.B, rows ? v.B : nullptr, act, a.T, kN, v.ldb, kN) ||
            !encode_matrix(&p.maps.C, rows ? v.C : nullptr, act, a.T, kN, v.ldc, kN))
            return MDRAFT_ERR_CUDA;
    }
    return launch_prefill<ML>(b, act, pl.form, call.stream) == cudaSuccess ? MDRAFT_OK : MDRAFT_ERR_CUDA;
}

// The one-kernel form (csrc/prefill_cluster.cu) of a call, or blocks = 0 where the plan above is the faster one.  Both are estimated:
//  - the one-kernel form takes kOne us and so much per block of a cluster, and per token of a chunk kLatency us plus kShare for every
//    further warp on a scheduler; short chunks of one block or two some 0.1 us a token more where they fill the machine; and 5 or 10 % more
//    where clusters of many or wide blocks fill SMs that they share: then some no longer fit beside the rest, most with another call's
//    blocks ahead of them (36 clusters of 7 blocks of 8 warps, 1128 channels x 1178 tokens: 28.3 us alone, 31.5 in a row; 24.7 by the rest of the estimate);
//  - the other takes kSplit + kSplitWork per token of work of a scheduler where it cuts sequences, kWhole + kWholeToken per token
//    of the longest where it does not.  That is good to 15 %, and high where a cut call fills an SM with blocks that finish together (24-token chunks of
//    1174 x 1112 18.7 us, estimated 21.8).
// So the one-kernel form has to promise 12 % less; 8 over several layers with A = powers and little work (57 calls that promise 8 to 12 %: 0.90 of the time in
// the mean, five lose 3 % and more); 16 where much work is cut (one layer, general A or fp32: of 94 such calls that promise 12 to 16 %, 29 lose 3 % and more; several
// layers, general A: 12 of 36; 8 layers of 3098 x 1016, fp32, A = powers: 190 us, in one kernel 233); 20 from sixteen sequences on, which the narrow form with four blocks to an SM serves better than estimated (20 x 1508 x 64, general A: 32.7 us, in
// one kernel 37.9); 25 where one layer's one sequence is long for its width (1500 x 1536: 26.8 us, in one kernel 29.6; 3925 x 368 28.5 and 34.4).
// It wins where the work is small: 256 x 64 fp32 9.2 -> 6.4 us, 256 x 768 bf16 12.3 -> 8.1, 1024 x 128 to 256 0.76 of the time; over 5170 calls that the rule
// gives to it (1 to 24 layers, 1 to 48 sequences of 2 to 5000 tokens, 32 to 1760 channels) it takes 0.78 of the other's time in the mean replayed from a
// graph, where 70 lose 3 to 15 %, and 0.70 called one after another, where 12 of 3089 lose 3 to 11 %.  (With 12, 20 and 25 % alone and no crowding 223 of 8727 lost 3 to 45 %
// replayed.  20 % wherever a cut call has much work, 14 elsewhere: 19 of 5709, but four times as many wins given up as losses saved.)  It loses where the work fills the machine, since its clusters
// leave a seventh of the SMs out and its channel groups are narrow: 1777 x 1536, general A, 35.5 against 41.4 at best, 4096 x 1536 52 against 77.
// A cluster reads its starting slot when it comes to run, by when another sequence's may have stored its final state, where the three kernels take the
// state and window that a cut sequence starts from ahead of the pass that stores.  The slots are on the device, so where several sequences have both and
// the plan cuts them (`shared`) the final states go through the workspace and a second kernel, for kDeliver us.
ClusterForm cluster_form(const mdraft_layer* L, int n_layers, int T, int n_seq, int max_seqlen, const mdraft_prefill_opts* opts, bool shared = false) {
    if (one_at_a_time(L) || (opts && (opts->chunk_len > 0 || opts->block_channels || opts->event_after_chunk_state || opts->event_after_carry_scan))) return {0, 0};
    constexpr double kOne = 4.1, kCluster = 0.6, kBlock = 0.13, kWarp = 0.15, kLatency[2] = {0.195, 0.275}, kShare[2] = {0.112, 0.167};
    constexpr double kSplit = 11.1, kSplitSeqs = 0.7, kSplitWork[2] = {0.166, 0.239}, kWhole = 3.3, kWholeToken = 0.104, kDeliver = 1.7;
    const int general = !(L->flags & MDRAFT_A_POWERS), sms = sm_count();
    const int64_t groups = (int64_t)n_layers * ((L->d_inner + kClusterCols - 1) / kClusterCols), clusters = groups * n_seq;
    const double work = (double)T * groups / (4 * sms);
    if (clusters > 8 * sms || (L->d_inner + kClusterCols - 1) / kClusterCols > 65535 || (int64_t)n_layers * n_seq > 65535) return {0, 0};
    ClusterForm best = {0, 0};
    double least = kSplit + work * kSplitWork[general] + (n_seq > 1 ? kSplitSeqs : 0.0);
    const double blocks = (double)n_layers * n_seq * ((L->d_inner + kPrefillThreads - 1) / kPrefillThreads), rounds = 1.2 * blocks / sms;
    const double whole = kWhole + max_seqlen * kWholeToken * (general ? kGeneralOne : 1.0) * (rounds > 1.0 ? rounds : 1.0);
    const bool much = least <= whole && (n_layers > 1 ? work > (general ? 80.0 : 200.0) : work > 40.0 && (general || L->act == MDRAFT_F32));
    const double margin = n_seq >= 16 ? 0.8 : n_seq * n_layers == 1 && work > 75.0 ? 0.75 : much ? 0.84 : n_layers > 1 && !general && work <= 120.0 ? 0.92 : 0.88;
    least = margin * (whole < least ? whole : least) - (shared ? kDeliver : 0.0);
    auto weigh = [&](int c, int w) {
        const int share = prefill_cluster_share(c, clusters);
        if (share * w > 16) return;   // the warps of an SM, 128 registers a thread
        const double busy = share * w > 4 ? share * w / 4.0 - 1.0 : 0.0;   // further warps on the fullest scheduler
        const double places = (double)clusters * c / (share * sms);            // of the SMs' room
        const int chunk = prefill_cluster_chunk(max_seqlen, c * w, !general);
        double t = kOne + (c > 1 ? kCluster : 0.0) + kBlock * c + kWarp * busy + chunk * (kLatency[general] + kShare[general] * busy);
        if (c <= 2 && places > 0.4) t += 0.1 * (places - 0.4) * (chunk < 16 ? chunk : 16);
        if (c >= 3 && share >= 2 && places > 0.72) t *= 1.0 + 0.05 * ((c >= 6) + (w == 8));
        if (t < least) { least = t; best = {c, w}; }
    };
    for (int w = 4; w <= kClusterMaxWarps; w *= 2)
        for (int c = 1; c <= kClusterMaxBlocks; ++c) weigh(c, w);
    return best;
}

template <int ML>
int run_prefill_cluster(const PrefillCall& call, const ClusterForm& form, const PrefillPlan* through, int32_t n_layers, const mdraft_layer* layers, const int32_t* layer_index, const mdraft_io* io) {
    ClusterBatch<ML> b;
    ClusterArgs& a = b.c;
    a.pool = PoolDev{};
    a.ssm_layer_stride = a.conv_layer_stride = 0;
    if (call.cache) {
        a.pool = pool_dev(call.cache, layers->act, 0);
        a.ssm_layer_stride = call.cache->ssm_layer_stride; a.conv_layer_stride = call.cache->conv_layer_stride;
    }
    a.n_layers = n_layers; a.d_inner = layers->d_inner; a.T = call.total_tokens; a.n_seq = call.n_seq;
    a.cu = call.cu_seqlens; a.init_slot = call.init_slot; a.final_slot = call.final_slot; a.dev_status = call.dev_status;
    a.ws_state = through ? reinterpret_cast<float*>(call.workspace + through->off_h0) : nullptr;
    a.ws_window = through ? call.workspace + through->off_conv : nullptr;
    a.ws_layer_bytes = through ? (int64_t)through->layer_bytes : 0;
    for (int32_t i = 0; i < n_layers; ++i) {
        const mdraft_io& v = io[i];
        b.l[i] = {layer_dev(layers + i), layer_index[i], v.x, v.z, v.dt, v.B, v.C, v.out, v.ldx, v.ldz, v.lddt, v.ldb, v.ldc, v.ldo};
    }
    return launch_prefill_cluster<ML>(b, layers->act, form, call.stream) == cudaSuccess ? MDRAFT_OK : MDRAFT_ERR_CUDA;
}

__global__ void classify_A_kernel(const float* A, int D, int N, int32_t* res) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= D * N) return;
    int d = i / N, n = i % N;
    float a0 = A[(size_t)d * N], a = A[i];
    if (a != (float)(n + 1) * a0) atomicOr(res + 0, 1);
    if (!(a <= 0.0f)) atomicOr(res + 1, 1);
}

}  // namespace

// The form of a call's first launch: 256 * blocks + warps of the one-kernel form, 0 for the plan's own kernels.  shared: the plan cuts its several sequences,
// which have both starting and final slots.  For the tests, which have to know what they run; no part of the interface.
extern "C" int32_t mdraft_internal_prefill_form(const mdraft_layer* layer, int32_t n_layers, int32_t total_tokens, int32_t n_seq, int32_t max_seqlen,
                                                int32_t shared) {
    if (check_layer(layer) != MDRAFT_OK || n_layers <= 0 || total_tokens <= 0 || n_seq <= 0 || max_seqlen <= 0) return 0;
    const int32_t most = prefill_most_layers(n_seq);
    const ClusterForm f = cluster_form(layer, n_layers < most ? n_layers : most, total_tokens, n_seq, max_seqlen < total_tokens ? max_seqlen : total_tokens, nullptr, shared != 0);
    return f.blocks * 256 + f.warps;
}

size_t mdraft::prefill_scratch_bytes(const mdraft_layer* layer, int32_t total_tokens, int32_t n_seq, int32_t max_seqlen, const mdraft_prefill_opts* opts,
                                     size_t available) {
    if (check_layer(layer) != MDRAFT_OK || total_tokens <= 0 || n_seq <= 0) return 0;
    if (max_seqlen < 1) max_seqlen = 1;
    const PrefillPlan pl = plan_prefill(layer, 1, total_tokens, n_seq, max_seqlen < total_tokens ? max_seqlen : total_tokens, opts, available);
    return pl.form.chunked ? pl.bytes : 0;
}

extern "C" {

const char* mdraft_status_string(int status) {
    switch (status) {
        case MDRAFT_OK: return "ok";
        case MDRAFT_ERR_INVALID_ARG: return "invalid argument";
        case MDRAFT_ERR_UNSUPPORTED: return "unsupported shape or dtype (need d_state=16, d_conv=4, d_inner%8==0, fp32/bf16)";
        case MDRAFT_ERR_MISALIGNED: return "pointer or stride not a multiple of 16 bytes";
        case MDRAFT_ERR_WORKSPACE: return "workspace missing or too small";
        case MDRAFT_ERR_CUDA: return "CUDA runtime error";
        default: return "unknown status";
    }
}

int mdraft_version(void) { return 100; }

size_t mdraft_prefill_workspace_bytes(const mdraft_layer* layer, int32_t total_tokens, int32_t n_seq, int32_t max_seqlen,
                                      const mdraft_prefill_opts* opts) {
    return mdraft_prefill_stack_workspace_bytes(layer, 1, total_tokens, n_seq, max_seqlen, opts);
}

size_t mdraft_prefill_stack_workspace_bytes(const mdraft_layer* layer, int32_t n_layers, int32_t total_tokens, int32_t n_seq,
                                            int32_t max_seqlen, const mdraft_prefill_opts* opts) {
    if (check_layer(layer) != MDRAFT_OK || n_layers <= 0 || total_tokens <= 0 || n_seq <= 0 || max_seqlen <= 0) return 0;
    // No sequence is longer than the whole batch: a looser static bound must not change the plan.
    if (max_seqlen > total_tokens) max_seqlen = total_tokens;
    size_t bytes = 0;  // the launches of one call share the workspace
    for_each_prefill_run(layer, n_layers, n_seq, [&](int32_t nl, int32_t) {
        const PrefillPlan pl = plan_prefill(layer, nl, total_tokens, n_seq, max_seqlen, opts, kAnyWorkspace);
        if ((n_layers == 1 || pl.form.chunked) && pl.bytes > bytes) bytes = pl.bytes;
    });
    return bytes;
}

int32_t mdraft_prefill_stack_launches(const mdraft_layer* layer, int32_t n_layers, int32_t total_tokens, int32_t n_seq,
                                      int32_t max_seqlen, const mdraft_prefill_opts* opts) {
    if (check_layer(layer) != MDRAFT_OK || n_layers <= 0 || total_tokens <= 0 || n_seq <= 0 || max_seqlen <= 0) return 0;
    if (max_seqlen > total_tokens) max_seqlen = total_tokens;
    int32_t n = 0;
    for_each_prefill_run(layer, n_layers, n_seq, [&](int32_t nl, int32_t times) {
        const bool one = cluster_form(layer, nl, total_tokens, n_seq, max_seqlen, opts).blocks > 0 || !plan_prefill(layer, nl, total_tokens, n_seq, max_seqlen, opts, kAnyWorkspace).form.chunked;
        n += times * (one ? 1 : (layer->flags & MDRAFT_CONV_ONLY) ? 2 : 3);
    });
    return n;
}

int mdraft_conv_scan_prefill(const mdraft_layer* layer, const mdraft_cache* cache, int32_t layer_index,
                             const void* x, int64_t ldx, const void* z, int64_t ldz, const void* dt, int64_t lddt,
                             const void* B, int64_t ldb, const void* C, int64_t ldc, void* out, int64_t ldo,
                             int32_t total_tokens, int32_t n_seq, int32_t max_seqlen, const int32_t* cu_seqlens,
                             const int32_t* init_slot, const int32_t* final_slot, void* workspace, size_t workspace_bytes,
                             const mdraft_prefill_opts* opts, int32_t* dev_status, void* stream) {
    const mdraft_io io = {x, z, dt, B, C, out, ldx, ldz, lddt, ldb, ldc, ldo};
    return mdraft_conv_scan_prefill_stack(1, layer, cache, &layer_index, &io, total_tokens, n_seq, max_seqlen, cu_seqlens, init_slot,
                                          final_slot, workspace, workspace_bytes, opts, dev_status, stream);
}

int mdraft_conv_scan_prefill_stack(int32_t n_layers, const mdraft_layer* layers, const mdraft_cache* cache, const int32_t* layer_index,
                                   const mdraft_io* io, int32_t total_tokens, int32_t n_seq, int32_t max_seqlen,
                                   const int32_t* cu_seqlens, const int32_t* init_slot, const int32_t* final_slot, void* workspace,
                                   size_t workspace_bytes, const mdraft_prefill_opts* opts, int32_t* dev_status, void* stream) {
    int rc = check_stack(n_layers, layers, layer_index, io);
    if (rc) return rc;
    if (total_tokens < 0 || n_seq < 0 || max_seqlen < 0) return MDRAFT_ERR_INVALID_ARG;
    if (opts) {
        if (opts->chunk_len < 0) return MDRAFT_ERR_INVALID_ARG;
        for (int i = 0; i < 2; ++i)
            if (opts->reserved[i]) return MDRAFT_ERR_INVALID_ARG;
        if (opts->block_channels != 0 && opts->block_channels != kPrefillThreads && opts->block_channels != kPrefillThreads * kPrefillWideBoxes)
            return MDRAFT_ERR_INVALID_ARG;
    }
    const int D = layers->d_inner, act = layers->act;
    if (init_slot || final_slot || cache) {
        for (int32_t i = 0; i < n_layers; ++i)
            if ((rc = check_cache(cache, D, act, layer_index[i]))) return rc;
    }
    if (n_seq == 0) return MDRAFT_OK;
    if (!cu_seqlens && n_seq != 1) return MDRAFT_ERR_INVALID_ARG;  // offsets may be omitted for a single sequence only
    const bool have_rows = total_tokens > 0;
    for (int32_t i = 0; i < n_layers; ++i)
        if ((rc = check_io(io[i], layers[i], have_rows))) return rc;
    // The same bound as in the workspace query: no sequence is longer than the whole batch.  A batch of empty
    // sequences therefore never takes the chunked path (and needs no workspace), whatever static bound was given.
    const int plan_tokens = total_tokens > 0 ? total_tokens : 1;
    if (max_seqlen > plan_tokens) max_seqlen = plan_tokens;
    if (max_seqlen < 1) max_seqlen = 1;

    const PrefillCall call = {cache, total_tokens, n_seq, cu_seqlens, init_slot, final_slot, static_cast<char*>(workspace), opts, dev_status,
                        static_cast<cudaStream_t>(stream)};
    // A sequence that is cut starts from what its slot held before the call, also where another stores there.
    auto shared_slots = [&](const PrefillPlan& pl) { return pl.form.chunked && n_seq > 1 && init_slot && final_slot; };
    for (int pass = 0; pass < 2; ++pass)  // every launch is checked before the first is made
        for (int32_t l0 = 0; l0 < n_layers;) {
            const int32_t nl = run_length(n_layers - l0, layers + l0, prefill_most_layers(n_seq));
            const PrefillPlan pl = plan_prefill(layers + l0, nl, plan_tokens, n_seq, max_seqlen, opts, workspace ? workspace_bytes : 0);
            if (pass == 0) {
                if (pl.n_chunks_bound > 65535 || (int64_t)nl * n_seq > 65535) return MDRAFT_ERR_UNSUPPORTED;
                if (pl.form.chunked) {
                    if (!workspace || workspace_bytes < pl.bytes) return MDRAFT_ERR_WORKSPACE;
                    if (reinterpret_cast<uintptr_t>(workspace) & 255u) return MDRAFT_ERR_MISALIGNED;
                }
            } else if (const ClusterForm cf = cluster_form(layers + l0, nl, plan_tokens, n_seq, max_seqlen, opts, shared_slots(pl)); cf.blocks > 0) {
                const PrefillPlan* through = shared_slots(pl) ? &pl : nullptr;
                const int r = nl == 1 ? run_prefill_cluster<1>(call, cf, through, nl, layers + l0, layer_index + l0, io + l0)
                                      : run_prefill_cluster<kClusterMaxLayers>(call, cf, through, nl, layers + l0, layer_index + l0, io + l0);
                if (r) return r;
            } else {
                const int r = nl == 1 ? run_prefill<1>(call, pl, nl, layers + l0, layer_index + l0, io + l0)
                                      : run_prefill<kPrefillMaxLayers>(call, pl, nl, layers + l0, layer_index + l0, io + l0);
                if (r) return r;
            }
            l0 += nl;
        }
    return MDRAFT_OK;
}

int mdraft_tree_step(const mdraft_layer* layer, const mdraft_cache* cache, int32_t layer_index, const void* x, int64_t ldx,
                     const void* z, int64_t ldz, const void* dt, int64_t lddt, const void* B, int64_t ldb, const void* C,
                     int64_t ldc, void* out, int64_t ldo, int32_t n_nodes, const int32_t* parent_slot,
                     const int32_t* node_slot, int32_t n_levels, const int32_t* level_offsets, int32_t* dev_status,
                     void* stream) {
    const mdraft_io io = {x, z, dt, B, C, out, ldx, ldz, lddt, ldb, ldc, ldo};
    return mdraft_tree_step_stack(1, layer, cache, &layer_index, &io, n_nodes, parent_slot, node_slot, n_levels, level_offsets, dev_status, stream);
}

int mdraft_tree_step_stack(int32_t n_layers, const mdraft_layer* layers, const mdraft_cache* cache, const int32_t* layer_index,
                           const mdraft_io* io, int32_t n_nodes, const int32_t* parent_slot, const int32_t* node_slot,
                           int32_t n_levels, const int32_t* level_offsets, int32_t* dev_status, void* stream) {
    int rc = check_stack(n_layers, layers, layer_index, io);
    if (rc) return rc;
    const int D = layers->d_inner, act = layers->act;
    for (int32_t i = 0; i < n_layers; ++i)
        if ((rc = check_cache(cache, D, act, layer_index[i]))) return rc;
    if (n_nodes < 0 || n_levels < 0) return MDRAFT_ERR_INVALID_ARG;
    if (n_nodes == 0) return MDRAFT_OK;
    if (!parent_slot || !node_slot) return MDRAFT_ERR_INVALID_ARG;
    if (!level_offsets && n_levels > 1) return MDRAFT_ERR_INVALID_ARG;
    if (level_offsets) {
        if (n_levels < 1 || level_offsets[0] != 0 || level_offsets[n_levels] != n_nodes) return MDRAFT_ERR_INVALID_ARG;
        for (int l = 0; l < n_levels; ++l)
            if (level_offsets[l + 1] < level_offsets[l]) return MDRAFT_ERR_INVALID_ARG;
    }
    for (int32_t i = 0; i < n_layers; ++i)
        if ((rc = check_io(io[i], layers[i], true))) return rc;

    TreeArgs a;
    a.pool = pool_dev(cache, act, 0);
    a.ssm_layer_stride = cache->ssm_layer_stride; a.conv_layer_stride = cache->conv_layer_stride;
    a.parent_slot = parent_slot; a.node_slot = node_slot; a.dev_status = dev_status;
    const int levels = level_offsets ? n_levels : 1;
    int launched = 0;  // an empty level launches nothing and must not count: the chaining rules go by kernels ahead
    for (int32_t l0 = 0; l0 < n_layers;) {
        const int32_t nl = run_length(n_layers - l0, layers + l0, kTreeMaxLayers);
        TreeLayers<kTreeMaxLayers> tl;
        for (int32_t i = 0; i < nl; ++i) {
            const mdraft_io& v = io[l0 + i];
            tl.l[i] = {layer_dev(layers + l0 + i), v.x, v.z, v.dt, v.B, v.C, v.out, v.ldx, v.ldz, v.lddt, v.ldb, v.ldc, v.ldo, layer_index[l0 + i]};
        }
        a.n_layers = nl;
        for (int l = 0; l < levels; ++l) {
            a.level_in_call = launched;
            a.lvl_begin = level_offsets ? level_offsets[l] : 0;
            a.lvl_end = level_offsets ? level_offsets[l + 1] : n_nodes;
            if (a.lvl_end == a.lvl_begin) continue;
            if (launch_tree_step(a, tl, act, static_cast<cudaStream_t>(stream)) != cudaSuccess) return MDRAFT_ERR_CUDA;
            ++launched;
        }
        l0 += nl;
    }
    return MDRAFT_OK;
}

int mdraft_tree_step_proj(const mdraft_layer* layer, const mdraft_cache* cache, int32_t layer_index,
                          const mdraft_select_proj* proj, const void* x, int64_t ldx, const void* z, int64_t ldz, void* out,
                          int64_t ldo, int32_t n_nodes, const int32_t* parent_slot, const int32_t* node_slot,
                          int32_t* dev_status, void* stream) {
    int rc = check_layer(layer);
    if (rc) return rc;
    if ((rc = check_cache(cache, layer->d_inner, layer->act, layer_index))) return rc;
    if (layer->flags & (MDRAFT_PRECONV | MDRAFT_CONV_ONLY)) return MDRAFT_ERR_INVALID_ARG;
    if (!proj || !proj->W_x || !proj->W_dt || n_nodes < 0) return MDRAFT_ERR_INVALID_ARG;
    if (!aligned16(proj->W_x) || !aligned16(proj->W_dt)) return MDRAFT_ERR_MISALIGNED;
    if (proj->dt_rank < 8 || proj->dt_rank > kProjMaxRank || (proj->dt_rank % 8) != 0) return MDRAFT_ERR_UNSUPPORTED;
    if (tree_proj_block_channels(layer->d_inner) == 0) return MDRAFT_ERR_UNSUPPORTED;
    if (proj->nodes_per_cluster != 0 && proj->nodes_per_cluster != 1 && proj->nodes_per_cluster != 2 && proj->nodes_per_cluster != 4)
        return MDRAFT_ERR_INVALID_ARG;
    if (n_nodes == 0) return MDRAFT_OK;
    if (!parent_slot || !node_slot) return MDRAFT_ERR_INVALID_ARG;
    const int D = layer->d_inner, act = layer->act;
    if ((rc = check_matrix(x, ldx, D, act, true))) return rc;
    if ((rc = check_matrix(z, ldz, D, act, true))) return rc;
    if ((rc = check_matrix(out, ldo, D, act, true))) return rc;

    TreeProjArgs a;
    a.L = layer_dev(layer);
    a.pool = pool_dev(cache, act, layer_index);
    a.x = x; a.z = z; a.out = out;
    a.ldx = ldx; a.ldz = ldz; a.ldo = ldo;
    a.W_x = proj->W_x; a.W_dt = proj->W_dt; a.dt_rank = proj->dt_rank; a.nodes_per_cluster = proj->nodes_per_cluster;
    a.parent_slot = parent_slot; a.node_slot = node_slot; a.n_nodes = n_nodes; a.chained = 0; a.most_shared = false; a.dev_status = dev_status;
    if (launch_tree_proj(a, act, static_cast<cudaStream_t>(stream)) != cudaSuccess) return MDRAFT_ERR_CUDA;
    return MDRAFT_OK;
}

int mdraft_block_generation(const mdraft_block_stack* stack, const mdraft_cache* cache, const int64_t* tokens, int32_t n_nodes,
                            const int32_t* parent_slot, const int32_t* node_slot, void* h, void* xz, void* y, void* logits, int64_t ldl,
                            int32_t* dev_status, void* stream) {
    if (!stack || stack->n_layers <= 0 || !stack->layers || !stack->W_in || !stack->W_x || !stack->W_dt || !stack->W_out || !stack->embed || !stack->W_lm)
        return MDRAFT_ERR_INVALID_ARG;
    if (n_nodes < 0) return MDRAFT_ERR_INVALID_ARG;
    const int D = stack->layers->d_inner, M = stack->d_model, R = stack->dt_rank;
    int rc;
    for (int32_t l = 0; l < stack->n_layers; ++l) {
        const mdraft_layer* L = stack->layers + l;
        if ((rc = check_layer(L))) return rc;
        if (L->d_inner != D || L->act != MDRAFT_BF16) return MDRAFT_ERR_UNSUPPORTED;
        if (L->flags & (MDRAFT_PRECONV | MDRAFT_CONV_ONLY)) return MDRAFT_ERR_INVALID_ARG;
        if ((rc = check_cache(cache, D, MDRAFT_BF16, l))) return rc;
        for (const void* w : {stack->W_in[l], stack->W_x[l], stack->W_dt[l], stack->W_out[l]}) {
            if (!w) return MDRAFT_ERR_INVALID_ARG;
            if (!aligned16(w)) return MDRAFT_ERR_MISALIGNED;
        }
    }
    if (M < 32 || M > kBlockMaxModel || M % 32 || D % 32 || D > kBlockMaxInner || stack->vocab < 8 || stack->vocab % 8 || R < 8 || R > kProjMaxRank ||
        R % 8 || tree_proj_block_channels(D) == 0 || n_nodes > kBlockMaxNodes)
        return MDRAFT_ERR_UNSUPPORTED;
    if (n_nodes == 0) return MDRAFT_OK;
    if (!tokens || !parent_slot || !node_slot || !h || !xz || !y || !logits || ldl < stack->vocab) return MDRAFT_ERR_INVALID_ARG;
    for (const void* q : {(const void*)h, (const void*)xz, (const void*)y, (const void*)logits, stack->embed, stack->W_lm})
        if (!aligned16(q)) return MDRAFT_ERR_MISALIGNED;
    if (ldl % 8) return MDRAFT_ERR_MISALIGNED;
    typedef __nv_bfloat16 bf;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    bf *hb = static_cast<bf*>(h), *xzb = static_cast<bf*>(xz), *yb = static_cast<bf*>(y);
    const ProductPlacement place = place_products(M, D, n_nodes);
    // The first kernel is an ordinary launch: everything ahead of the call is complete before a kernel of the call reads
    // a parent's state, which no other kernel of the call writes.  Each later kernel may start while the one ahead runs.
    cudaError_t e = launch_embed(tokens, static_cast<const bf*>(stack->embed), hb, n_nodes, M, stack->vocab, dev_status, st);
    for (int32_t l = 0; l < stack->n_layers && e == cudaSuccess; ++l) {
        e = launch_small_linear({hb, static_cast<const bf*>(stack->W_in[l]), nullptr, xzb, 2 * (int64_t)D, 2 * (int64_t)D, n_nodes, 2 * D, M, dev_status, false, place.in_alone, stack->eps}, st);
        if (e != cudaSuccess) break;
        TreeProjArgs a;
        a.L = layer_dev(stack->layers + l);
        a.pool = pool_dev(cache, MDRAFT_BF16, l);
        a.x = xzb; a.z = xzb + D; a.out = yb;
        a.ldx = a.ldz = 2 * (int64_t)D; a.ldo = D;
        a.W_x = stack->W_x[l]; a.W_dt = stack->W_dt[l]; a.dt_rank = R; a.nodes_per_cluster = 0;
        a.parent_slot = parent_slot; a.node_slot = node_slot; a.n_nodes = n_nodes; a.chained = 1; a.most_shared = place.step_split; a.dev_status = dev_status;
        if ((e = launch_tree_proj(a, MDRAFT_BF16, st)) != cudaSuccess) break;
        e = launch_small_linear({yb, static_cast<const bf*>(stack->W_out[l]), hb, hb, M, M, n_nodes, M, D, dev_status, place.out_late, place.out_alone, -1.0f}, st);
    }
    if (e == cudaSuccess)
        e = launch_small_linear({hb, static_cast<const bf*>(stack->W_lm), nullptr, static_cast<bf*>(logits), stack->vocab, ldl, n_nodes, stack->vocab, M, dev_status, false, false, stack->eps}, st);
    return e == cudaSuccess ? MDRAFT_OK : MDRAFT_ERR_CUDA;
}

int mdraft_state_commit(const mdraft_cache* cache, int32_t d_inner, int32_t d_state, int32_t d_conv, int32_t act,
                        int32_t n_commit, const int32_t* src_slot, const int32_t* dst_slot, int32_t* dev_status,
                        void* stream) {
    if (d_inner <= 0 || n_commit < 0) return MDRAFT_ERR_INVALID_ARG;
    if ((d_state != kN && d_state != kSsdN) || d_conv != kW || (d_inner % 8) != 0 || (act != MDRAFT_F32 && act != MDRAFT_BF16)) return MDRAFT_ERR_UNSUPPORTED;
    int rc = check_cache(cache, d_inner, act, 0, d_state);
    if (rc) return rc;
    if (n_commit == 0) return MDRAFT_OK;
    if (!src_slot || !dst_slot) return MDRAFT_ERR_INVALID_ARG;
    const int64_t es = (int64_t)elem_size(act);
    CommitArgs a;
    a.ssm = reinterpret_cast<char*>(cache->ssm);
    a.conv = static_cast<char*>(cache->conv);
    a.ssm_layer_bytes = cache->ssm_layer_stride * 4; a.ssm_slot_bytes_stride = cache->ssm_slot_stride * 4;
    a.conv_layer_bytes = cache->conv_layer_stride * es; a.conv_slot_bytes_stride = cache->conv_slot_stride * es;
    a.ssm_bytes = (int64_t)d_inner * d_state * 4; a.conv_bytes = (int64_t)(kW - 1) * d_inner * es;
    a.n_layers = cache->n_layers; a.n_slots = cache->n_slots; a.dev_status = dev_status;
    if (a.n_layers > 65535) return MDRAFT_ERR_UNSUPPORTED;
    for (int off = 0; off < n_commit; off += 65535) {
        a.n_commit = n_commit - off < 65535 ? n_commit - off : 65535;
        a.src_slot = src_slot + off; a.dst_slot = dst_slot + off;
        if (launch_commit(a, static_cast<cudaStream_t>(stream)) != cudaSuccess) return MDRAFT_ERR_CUDA;
    }
    return MDRAFT_OK;
}

int mdraft_classify_A(const float* A, int32_t d_inner, int32_t d_state, int32_t* scratch, int32_t* is_powers,
                      int32_t* is_nonpositive, void* stream) {
    if (!A || !scratch || !is_powers || d_inner <= 0 || d_state <= 0) return MDRAFT_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(scratch, 0, 2 * sizeof(int32_t), st) != cudaSuccess) return MDRAFT_ERR_CUDA;
    const int n = d_inner * d_state;
    classify_A_kernel<<<(n + 255) / 256, 256, 0, st>>>(A, d_inner, d_state, scratch);
    int32_t host[2] = {1, 1};
    if (cudaMemcpyAsync(host, scratch, sizeof(host), cudaMemcpyDeviceToHost, st) != cudaSuccess) return MDRAFT_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return MDRAFT_ERR_CUDA;
    *is_powers = host[0] == 0;
    if (is_nonpositive) *is_nonpositive = host[1] == 0;
    return MDRAFT_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------------- SSD layer
namespace {

int check_ssd_layer(const mdraft_ssd_layer* L) {
    if (!L || !L->A || !L->conv_w) return MDRAFT_ERR_INVALID_ARG;
    if (L->d_inner <= 0) return MDRAFT_ERR_INVALID_ARG;
    if (L->headdim != kSsdP || L->d_state != kSsdN || L->d_conv != kW || (L->d_inner % kSsdP) != 0 || L->act != MDRAFT_BF16)
        return MDRAFT_ERR_UNSUPPORTED;
    if (L->flags & ~(uint32_t)MDRAFT_DT_SOFTPLUS) return MDRAFT_ERR_INVALID_ARG;
    if (!aligned16(L->conv_w)) return MDRAFT_ERR_MISALIGNED;
    return MDRAFT_OK;
}

SsdLayerDev ssd_layer_dev(const mdraft_ssd_layer* L) {
    SsdLayerDev d;
    d.A = L->A; d.D = L->D; d.conv_w = L->conv_w; d.conv_b = L->conv_b; d.dt_bias = L->dt_bias;
    d.d_inner = L->d_inner; d.n_heads = L->d_inner / L->headdim; d.flags = L->flags;
    return d;
}

struct SsdPlan {
    int n_chunks_bound;
    size_t off_S, off_decay, off_hin, off_xd, off_u, off_csl, bytes;
};

SsdPlan plan_ssd(const mdraft_ssd_layer* L, int T, int n_seq) {
    SsdPlan pl;
    const size_t H = (size_t)(L->d_inner / L->headdim);
    pl.n_chunks_bound = n_seq + T / kSsdQ;
    const size_t per_chunk = H * kSsdP * kSsdN;
    pl.off_S = 0;
    pl.off_decay = align_up(pl.off_S + (size_t)pl.n_chunks_bound * per_chunk * sizeof(float), 256);
    pl.off_hin = align_up(pl.off_decay + (size_t)pl.n_chunks_bound * H * sizeof(float), 256);
    pl.off_xd = align_up(pl.off_hin + (size_t)pl.n_chunks_bound * per_chunk * 2 * 2, 256);   // bf16 value + bf16 remainder
    pl.off_u = align_up(pl.off_xd + (size_t)pl.n_chunks_bound * H * (kSsdP / 8) * (kSsdQ * 16 + 16), 256);
    pl.off_csl = align_up(pl.off_u + (size_t)T * L->d_inner * 2, 256);
    pl.bytes = align_up(pl.off_csl + (size_t)pl.n_chunks_bound * H * kSsdQ * sizeof(float), 256);
    return pl;
}

// Descriptor of a (rows x cols) row-major bf16 matrix read in boxes of box_cols x 128 rows.
bool encode_ssd_matrix(CUtensorMap* m, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_cols) {
    PFN_cuTensorMapEncodeTiled enc = tensor_map_encoder();
    if (!enc) return false;
    cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t gstride[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)kSsdQ};
    cuuint32_t estride[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Descriptor of a (rows x 128) row-major bf16 matrix read in boxes of 64 columns x 128 rows that land in shared memory as
// rows of 128 bytes, 16-byte units XOR-ed with the row index (the tensor core's 128-byte-swizzled K-major operand layout).
bool encode_ssd_swizzled(CUtensorMap* m, const void* base, int64_t rows, int64_t ld) {
    PFN_cuTensorMapEncodeTiled enc = tensor_map_encoder();
    if (!enc) return false;
    cuuint64_t gdim[2] = {(cuuint64_t)kSsdN, (cuuint64_t)rows};
    cuuint64_t gstride[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)kSsdQ};
    cuuint32_t estride[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

extern "C" {

size_t mdraft_ssd_prefill_workspace_bytes(const mdraft_ssd_layer* layer, int32_t total_tokens, int32_t n_seq) {
    if (check_ssd_layer(layer) != MDRAFT_OK || total_tokens <= 0 || n_seq <= 0) return 0;
    return plan_ssd(layer, total_tokens, n_seq).bytes;
}

int mdraft_ssd_prefill(const mdraft_ssd_layer* layer, const mdraft_cache* cache, int32_t layer_index, const void* x, int64_t ldx,
                       const void* z, int64_t ldz, const void* dt, int64_t lddt, const void* B, int64_t ldb, const void* C,
                       int64_t ldc, void* out, int64_t ldo, int32_t total_tokens, int32_t n_seq, const int32_t* cu_seqlens,
                       const int32_t* init_slot, const int32_t* final_slot, void* workspace, size_t workspace_bytes,
                       int32_t* dev_status, void* stream) {
    int rc = check_ssd_layer(layer);
    if (rc) return rc;
    if (total_tokens < 0 || n_seq < 0) return MDRAFT_ERR_INVALID_ARG;
    if (init_slot || final_slot || cache) {
        rc = check_cache(cache, layer->d_inner, layer->act, layer_index, kSsdN);
        if (rc) return rc;
    }
    if (n_seq == 0) return MDRAFT_OK;
    if (!cu_seqlens && n_seq != 1) return MDRAFT_ERR_INVALID_ARG;
    const int D = layer->d_inner, H = D / layer->headdim;
    const bool have_rows = total_tokens > 0;
    if ((rc = check_matrix(x, ldx, D, MDRAFT_BF16, have_rows))) return rc;
    if ((rc = check_matrix(z, ldz, D, MDRAFT_BF16, have_rows))) return rc;
    if ((rc = check_matrix(out, ldo, D, MDRAFT_BF16, have_rows))) return rc;
    if ((rc = check_matrix(B, ldb, kSsdN, MDRAFT_BF16, have_rows))) return rc;
    if ((rc = check_matrix(C, ldc, kSsdN, MDRAFT_BF16, have_rows))) return rc;
    if (have_rows && (!dt || lddt < H)) return MDRAFT_ERR_INVALID_ARG;
    const SsdPlan pl = plan_ssd(layer, have_rows ? total_tokens : 1, n_seq);
    if (!workspace || workspace_bytes < pl.bytes) return MDRAFT_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(workspace) & 255u) return MDRAFT_ERR_MISALIGNED;
    if (pl.n_chunks_bound > 65535) return MDRAFT_ERR_UNSUPPORTED;

    SsdPrefillArgs a;
    a.L = ssd_layer_dev(layer);
    if (cache) a.pool = pool_dev(cache, MDRAFT_BF16, layer_index);
    else { a.pool.ssm = nullptr; a.pool.conv = nullptr; a.pool.ssm_slot_stride = 0; a.pool.conv_slot_stride = 0; a.pool.n_slots = 0; }
    a.x = static_cast<const __nv_bfloat16*>(x); a.z = static_cast<const __nv_bfloat16*>(z); a.dt = static_cast<const __nv_bfloat16*>(dt);
    a.B = static_cast<const __nv_bfloat16*>(B); a.C = static_cast<const __nv_bfloat16*>(C); a.out = static_cast<__nv_bfloat16*>(out);
    a.ldx = ldx; a.ldz = ldz; a.lddt = lddt; a.ldb = ldb; a.ldc = ldc; a.ldo = ldo;
    a.T = total_tokens; a.n_seq = n_seq; a.n_chunks_bound = pl.n_chunks_bound;
    a.cu = cu_seqlens; a.init_slot = init_slot; a.final_slot = final_slot;
    char* ws = static_cast<char*>(workspace);
    a.ws_S = reinterpret_cast<float*>(ws + pl.off_S);
    a.ws_decay = reinterpret_cast<float*>(ws + pl.off_decay);
    a.ws_hin = reinterpret_cast<__nv_bfloat16*>(ws + pl.off_hin);
    a.ws_xd = reinterpret_cast<__nv_bfloat16*>(ws + pl.off_xd);
    a.ws_u = reinterpret_cast<__nv_bfloat16*>(ws + pl.off_u);
    a.ws_csl = reinterpret_cast<float*>(ws + pl.off_csl);
    a.dev_status = dev_status;
    SsdMaps maps;
    memset(&maps, 0, sizeof(maps));
    if (have_rows) {
        if (!encode_ssd_matrix(&maps.x, x, total_tokens, D, ldx, kSsdP) || !encode_ssd_matrix(&maps.z, z, total_tokens, D, ldz, kSsdP) ||
            !encode_ssd_swizzled(&maps.Bs, B, total_tokens, ldb) ||
            !encode_ssd_swizzled(&maps.Cs, C, total_tokens, ldc))
            return MDRAFT_ERR_CUDA;
    }
    return launch_ssd_prefill(a, maps, static_cast<cudaStream_t>(stream)) == cudaSuccess ? MDRAFT_OK : MDRAFT_ERR_CUDA;
}

int mdraft_ssd_tree_step(const mdraft_ssd_layer* layer, const mdraft_cache* cache, int32_t layer_index, const void* x, int64_t ldx,
                         const void* z, int64_t ldz, const void* dt, int64_t lddt, const void* B, int64_t ldb, const void* C,
                         int64_t ldc, void* out, int64_t ldo, int32_t n_nodes, const int32_t* parent_slot, const int32_t* node_slot,
                         int32_t n_levels, const int32_t* level_offsets, int32_t* dev_status, void* stream) {
    int rc = check_ssd_layer(layer);
    if (rc) return rc;
    if ((rc = check_cache(cache, layer->d_inner, layer->act, layer_index, kSsdN))) return rc;
    if (n_nodes < 0 || n_levels < 0) return MDRAFT_ERR_INVALID_ARG;
    if (n_nodes == 0) return MDRAFT_OK;
    if (!parent_slot || !node_slot) return MDRAFT_ERR_INVALID_ARG;
    if (!level_offsets && n_levels > 1) return MDRAFT_ERR_INVALID_ARG;
    if (level_offsets) {
        if (n_levels < 1 || level_offsets[0] != 0 || level_offsets[n_levels] != n_nodes) return MDRAFT_ERR_INVALID_ARG;
        for (int l = 0; l < n_levels; ++l)
            if (level_offsets[l + 1] < level_offsets[l]) return MDRAFT_ERR_INVALID_ARG;
    }
    const int D = layer->d_inner, H = D / layer->headdim;
    if ((rc = check_matrix(x, ldx, D, MDRAFT_BF16, true))) return rc;
    if ((rc = check_matrix(z, ldz, D, MDRAFT_BF16, true))) return rc;
    if ((rc = check_matrix(out, ldo, D, MDRAFT_BF16, true))) return rc;
    if ((rc = check_matrix(B, ldb, kSsdN, MDRAFT_BF16, true))) return rc;
    if ((rc = check_matrix(C, ldc, kSsdN, MDRAFT_BF16, true))) return rc;
    if (!dt || lddt < H) return MDRAFT_ERR_INVALID_ARG;
    SsdStepArgs a;
    a.L = ssd_layer_dev(layer);
    a.pool = pool_dev(cache, MDRAFT_BF16, layer_index);
    a.x = static_cast<const __nv_bfloat16*>(x); a.z = static_cast<const __nv_bfloat16*>(z); a.dt = static_cast<const __nv_bfloat16*>(dt);
    a.B = static_cast<const __nv_bfloat16*>(B); a.C = static_cast<const __nv_bfloat16*>(C); a.out = static_cast<__nv_bfloat16*>(out);
    a.ldx = ldx; a.ldz = ldz; a.lddt = lddt; a.ldb = ldb; a.ldc = ldc; a.ldo = ldo;
    a.parent_slot = parent_slot; a.node_slot = node_slot; a.dev_status = dev_status;
    const int levels = level_offsets ? n_levels : 1;
    a.level_in_call = 0;
    for (int l = 0; l < levels; ++l) {
        a.lvl_begin = level_offsets ? level_offsets[l] : 0;
        a.lvl_end = level_offsets ? level_offsets[l + 1] : n_nodes;
        if (a.lvl_end == a.lvl_begin) continue;
        if (launch_ssd_step(a, static_cast<cudaStream_t>(stream)) != cudaSuccess) return MDRAFT_ERR_CUDA;
        ++a.level_in_call;
    }
    return MDRAFT_OK;
}

}  // extern "C"
