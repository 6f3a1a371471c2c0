// Host side of the C ABI: argument validation, channel-map compilation, workspace handling
// and the dispatch by M between the decode, prefill and generic kernels.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <mutex>

#include "common.cuh"

using namespace uniql;

namespace {

std::atomic<int> g_path{UNIQL_PATH_AUTO};

// name, environment variable read once at load, default
struct OptDesc { const char* name; const char* env; int dflt; };
const OptDesc kOpts[kOptCount] = {
    {"pdl", "UNIQL_PDL", 1},                            // programmatic stream serialization (decode and tensor-core launches)
    {"decode_kp", "UNIQL_DECODE_KP", 0},                // groups of blocks over the input channels (0: automatic)
    {"decode_rp", "UNIQL_DECODE_RP", 0},                // blocks per group (0: one per SM)
    {"decode_stages", "UNIQL_DECODE_STAGES", 0},        // ring stages (0: automatic)
    {"decode_narrow", "UNIQL_DECODE_NARROW", -1},       // narrow tiles: -1 automatic, 0 off, 1 on
    {"decode_xstream", "UNIQL_DECODE_XSTREAM", -1},     // streamed activations: -1 automatic, 0 off, 1 on
    {"decode_xcluster", "UNIQL_DECODE_XCLUSTER", -1},   // shared staging in clusters of two: -1 automatic, 0 off, 1 on
    {"decode_i8", "UNIQL_DECODE_I8", 1},                // integer path (0: fp16 MMAs)
    {"decode_split_batch", "UNIQL_DECODE_SPLIT_BATCH", 2},   // batches of 9..16: one streamed launch where it applies
    {"prefill_grid", "UNIQL_PREFILL_GRID", 0},          // blocks of the tensor-core kernel (0: one per SM)
    {"prefill_convert", "UNIQL_PREFILL_CONVERT_IN_KERNEL", 0},   // 1: bf16 tiles converted inside the kernel
    {"prefill_streamk", "UNIQL_PREFILL_STREAMK", -1},   // split tiles: -1 automatic, 0 never, 1 always (a slot per part), 2 always (one sum per tile), 3 pairs of blocks
    {"prefill_dual", "UNIQL_PREFILL_DUAL", -1},         // tiles of 512 tokens on both accumulators: -1 by cost, 0 never, 1 always (2 / 3: without / with half tiles)
    {"prefill_helpers", "UNIQL_PREFILL_HELPERS", 1},    // de-quantiser warps share the epilogue of a block's last tile
    {"prefill_pair", "UNIQL_PREFILL_PAIR", -1},         // block pairs (cta_group::2): -1 by cost, 0 never, 1 / 2 always, with 256 / 512 tokens per tile, 3 by cost and refused at launch
    {"gemv_first", "UNIQL_GEMV_FIRST", 0},              // 1: the streaming kernel wherever it applies (M <= 4)
    {"gemv_depth", "UNIQL_GEMV_DEPTH", 0},              // ring slots per warp of the streaming kernel (0: automatic)
    {"wait_shift", "UNIQL_WAIT_SHIFT", 0},              // bounded device waits: limits divided by 2^shift (tests)
};
std::atomic<int> g_opt[kOptCount];
const bool g_opt_init = [] {
  for (int i = 0; i < kOptCount; ++i) {
    const char* e = getenv(kOpts[i].env);
    g_opt[i].store(e ? atoi(e) : kOpts[i].dflt);
  }
  return true;
}();

constexpr int kMaxDevices = 64;
constexpr size_t kLibWorkspaceBytes = (size_t)192 << 20;
void* g_ws[kMaxDevices] = {nullptr};
std::mutex g_ws_mutex;

// Per-device library workspace, allocated (and its counters zeroed) at first use.
int lib_workspace(void** ws, size_t* bytes, cudaStream_t stream) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return UNIQL_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_ws_mutex);
  if (!g_ws[dev]) {
    void* p = nullptr;
    if (cudaMalloc(&p, kLibWorkspaceBytes) != cudaSuccess) { cudaGetLastError(); return UNIQL_ERR_CUDA; }
    if (cudaMemset(p, 0, kLibWorkspaceBytes) != cudaSuccess) { cudaFree(p); return UNIQL_ERR_CUDA; }
    g_ws[dev] = p;
  }
  (void)stream;
  *ws = g_ws[dev];
  *bytes = kLibWorkspaceBytes;
  return UNIQL_OK;
}

// Validate a caller map against a dimension of size D and compile it.
int compile_map(const uniql_chanmap* src, int k_lead, int D, ChanMap* out) {
  memset(out, 0, sizeof(*out));
  if (!src) {
    if (k_lead <= 0 || k_lead > D) return UNIQL_ERR_SHAPE;
    out->n_fam = 1;
    out->fam[0] = Fam{0, k_lead, k_lead, 1};
    out->base[0] = 0;
    out->total = k_lead;
    return UNIQL_OK;
  }
  if (src->n_fam < 1 || src->n_fam > kMaxFam) return UNIQL_ERR_SHAPE;
  int64_t prev_end = 0, total = 0;
  for (int f = 0; f < src->n_fam; ++f) {
    const uniql_family& a = src->fam[f];
    if (a.start < 0 || a.keep <= 0 || a.count <= 0 || a.period <= 0) return UNIQL_ERR_SHAPE;
    if (a.count > 1 && a.period < a.keep) return UNIQL_ERR_SHAPE;
    int64_t end = (int64_t)a.start + (int64_t)(a.count - 1) * a.period + a.keep;
    if (a.start < prev_end || end > D) return UNIQL_ERR_SHAPE;
    prev_end = end;
    out->fam[f] = Fam{a.start, a.period, a.keep, a.count};
    out->base[f] = (int)total;
    total += (int64_t)a.keep * a.count;
  }
  if (total > D) return UNIQL_ERR_SHAPE;
  out->n_fam = src->n_fam;
  out->total = (int)total;
  return UNIQL_OK;
}

int check_common(const void* x, int ldx, int dt, int M, int K) {
  if (!x) return UNIQL_ERR_NULL;
  if (dt != UNIQL_F16 && dt != UNIQL_BF16) return UNIQL_ERR_DTYPE;
  if (M < 1 || K < kGroup || (K % kGroup) != 0 || ldx < 1) return UNIQL_ERR_SHAPE;
  if (((uintptr_t)x) & 1) return UNIQL_ERR_ALIGN;
  return UNIQL_OK;
}

int check_weight(const uint8_t* w, const void* s, const void* z, int N) {
  if (!w || !s || !z) return UNIQL_ERR_NULL;
  if (N < 1) return UNIQL_ERR_SHAPE;
  if ((((uintptr_t)w) & 15) || (((uintptr_t)s) & 1) || (((uintptr_t)z) & 1)) return UNIQL_ERR_ALIGN;
  return UNIQL_OK;
}

// The activations re-laid so that the fast kernels can read them: one input family whose kept blocks (or whose row
// pitch / base address) are not on 16-byte boundaries becomes the same family with every block padded to a multiple
// of 8 channels, the padding zero (the extra channels then meet real weights with zero activations).  Fills `q` with
// the parameters of the re-laid problem (x still to be set) and returns the padded block size, or 0 when the map
// does not allow it.
int relay_candidate(const Params& p, Params* q) {
  if (p.imap.n_fam != 1) return 0;
  const Fam& a = p.imap.fam[0];
  const int keep8 = (a.keep + 7) / 8 * 8;
  if ((a.start % 8) != 0) return 0;
  if (a.count > 1 && ((a.period % 8) != 0 || keep8 > a.period)) return 0;
  if (a.count == 1 && a.start + keep8 > p.K) return 0;
  *q = p;
  q->imap.fam[0].keep = keep8;
  q->imap.total = keep8 * a.count;
  q->imap.base[0] = 0;
  q->k_in = q->imap.total;
  q->ldx = q->imap.total;
  q->x = reinterpret_cast<const void*>((uintptr_t)256);     // (aligned as the workspace region will be)
  return keep8;
}

int dispatch_as(const Params& p_in, int path, void* workspace, size_t ws_bytes, void* stream) {
  LaunchCfg cfg{workspace, ws_bytes, (cudaStream_t)stream};
  Params p = p_in;
  // The rows of a decode launch: option "decode_split_batch" (or streaming turned off) runs nine to sixteen rows as two
  // launches, and what those can take is asked for them (five to eight rows need activations on 8-channel boundaries).
  const bool streams = opt(kOptDecodeSplitBatch) == 2 && opt(kOptDecodeI8) != 0 && opt(kOptDecodeXstream) != 0;
  const bool halves = p.M > 8 && p.M <= 16 && !streams && opt(kOptDecodeSplitBatch) != 0;
  auto as_launched = [&](const Params& a, int (*holds)(const Params&)) {
    if (!halves) return holds(a) != 0;
    Params q = a;
    q.M = (q.M + 1) / 2;
    return holds(q) != 0;
  };
  auto decodes = [&](const Params& a) { return a.M <= 16 && as_launched(a, decode_supported); };
  auto on_integers = [&](const Params& a) { return as_launched(a, decode_integer_path); };
  bool dec_ok = decodes(p);
  // every batch the decode kernel does not take (more than 16 rows) goes to the tensor cores when the maps
  // allow it: at 17..63 rows the generic kernel measured 13 to 26 times slower (930 us against 71 us for the
  // Llama-3-8B gate|up at M = 17)
  // (fp16 up to 128 rows: the batch kernel also takes heads that keep 4 (mod 8) channels, where the workspace has its header: such a
  //  call is re-laid with more room and ran on the generic kernel, which needs none, with less)
  auto on_tensor_cores = [&](const Params& a) {
    return prefill_supported(a) != 0 || (a.dt == UNIQL_F16 && batch_supported(a) != 0 &&
                                         (!cfg.workspace || cfg.ws_bytes >= decode_workspace_header_bytes()));
  };
  bool pre_ok = on_tensor_cores(p);
  // The streaming kernel (one to four rows): where it is asked for, and where the decode kernel's integer path cannot run
  // (scales on 8- but not 16-byte boundaries).
  bool gv = path == UNIQL_PATH_GEMV || (path == UNIQL_PATH_AUTO && gemv_supported(p) && opt(kOptGemvFirst) == 1);
  const bool gv_else = path == UNIQL_PATH_AUTO && !gv && gemv_supported(p) && !(dec_ok && on_integers(p));
  bool relaid = false;
  // What misses a fast kernel only because of where its activations lie (above 16 rows blocks of 108 or 84 channels, at
  // decode sizes blocks that are no multiple of 4, an odd row pitch) gets them re-laid in the workspace by a small kernel
  // in front.
  if (!gv && path != UNIQL_PATH_GENERIC) {
    bool decode_size = p.M <= 16 && path != UNIQL_PATH_PREFILL;
    Params q;
    int keep8 = 0;
    // (bf16 at decode sizes that the integer path cannot take even re-laid: the tensor cores, as larger batches)
    if (decode_size && p.dt != UNIQL_F16 && path == UNIQL_PATH_AUTO && !dec_ok &&
        !(relay_candidate(p, &q) != 0 && decodes(q)))
      decode_size = false;
    const bool slow = decode_size ? !(dec_ok && on_integers(p)) : !pre_ok;
    if (slow && path != (decode_size ? UNIQL_PATH_PREFILL : UNIQL_PATH_DECODE) && (keep8 = relay_candidate(p, &q)) != 0 &&
        (decode_size ? (decodes(q) && on_integers(q)) : prefill_supported(q))) {
      if (!cfg.workspace) {
        int rc = lib_workspace(&cfg.workspace, &cfg.ws_bytes, cfg.stream);
        if (rc != UNIQL_OK) return rc;
      }
      const size_t floor_bytes = decode_size ? decode_workspace_bytes(p.M, p.K, 1) : decode_workspace_header_bytes();
      // (tensor cores: rows of whole 128-byte lines, as launch_planned() has them, where there is room)
      const int lines = (q.ldx + 63) / 64 * 64;
      if (!decode_size && cfg.ws_bytes >= (size_t)p.M * (size_t)lines * 2 + 255 + floor_bytes + 256) q.ldx = lines;
      const size_t bytes = (((size_t)p.M * (size_t)q.ldx * 2) + 255) & ~(size_t)255;
      if (cfg.ws_bytes >= bytes + floor_bytes + 256) {
        // the copy lives at the end of the workspace; the kernels get what lies before it
        const size_t off = (cfg.ws_bytes - bytes) & ~(size_t)255;
        void* xr = reinterpret_cast<unsigned char*>(cfg.workspace) + off;
        const Fam& a = p.imap.fam[0];
        // (bf16 above 16 rows goes to the tensor cores, whose operands are fp16: converted on the way)
        const bool to_f16 = p.dt == UNIQL_BF16 && p.M > 16 && opt(kOptPrefillConvert) != 1;
        int rc = launch_relay_x(p.x, p.ldx, p.M, a.count, a.keep, keep8, xr, q.ldx, to_f16, p.M > 16 && p.M <= 128, cfg.stream);
        if (rc != UNIQL_OK) return rc;
        q.x = xr;
        q.x_f16 = to_f16 ? 1 : 0;
        p = q;
        relaid = true;
        cfg.ws_bytes = off;
        dec_ok = decodes(p);
        pre_ok = on_tensor_cores(p);
      }
    }
  }
  if (gv_else && !relaid) gv = true;
  // An odd number of groups: the decode kernel or, above sixteen rows, the batch kernel on a copy of the scales and zero-points
  // with rows padded to eight groups, a sixteenth of the codes' bytes (short rows more: all of a half for one group).  On single
  // blocks of the tensor-core kernel, which takes what stays here, 10192 x 10624 at two rows is 52 us where its bytes take 8 (here
  // 18).  Not under options that run a batch as two halves.
  if (path == UNIQL_PATH_AUTO && !gv && !dec_ok && p.M <= 128 && !halves && (p.K / kGroup) % 2 != 0) {
    Params q = p;
    const int G = p.K / kGroup;
    q.sz_pitch = (G + 7) / 8 * 8;
    size_t at[kMaxJobs + 1] = {0};
    int rows[kMaxJobs] = {0}, n_total = 0;
    bool small = true;
    int64_t codes = 0;
    for (int j = 0; j < p.n_jobs; ++j) {                     // (rows up to the last kept one)
      const Fam& f = p.job[j].omap.fam[p.job[j].omap.n_fam - 1];
      rows[j] = f.start + (f.count - 1) * f.period + f.keep;
      n_total += p.job[j].k_out;
      codes += (int64_t)p.job[j].k_out * p.k_in;
      small = small && (int64_t)rows[j] * (q.sz_pitch / 8) < (1 << 30);
      at[j + 1] = at[j] + (((size_t)rows[j] * q.sz_pitch * 4 + 255) & ~(size_t)255);
      q.job[j].scales = q.job[j].zeros = nullptr;            // (aligned as the copies will be)
    }
    // A single block walks its tile's groups one by one and the copy is a launch of its own (2 us), so few groups stay unless there
    // are tiles for several rounds.  Single blocks -> decode kernel at one / eight rows: 512 x 384 5.9 -> 6.9 / 5.9 -> 6.8 us, 2048 x 384
    // 6.2 -> 7.0 / 7.1, 9216 x 384 6.7 -> 5.9 / 8.5, 14336 x 384 7.8 -> 6.3 / 9.1, 32768 x 384 11.2 -> 8.3 / 11.3, 128 x 640 7.7 -> 5.9 / 8.0 -> 7.0.
    // Nine to sixteen rows have a second kernel in front, which quantises the activations: at nine rows half a million codes
    // 9.2 -> 10.2 us, 9 million 11.5 -> 11.6, 6144 x 1664 13.3 -> 10.4, 17 million 18.4 -> 14.5; with nine groups 9216 / 16384 / 28672 rows
    // 11.7 -> 11.5 / 13.5 -> 14.3 / 33.0 -> 19.6; 32768 x 384 11.5 -> 15.5, x 640 14.9 -> 16.7.
    const int groups = (p.k_in + kGroup - 1) / kGroup;
    // (a copy per matrix: q|k|v of 640 channels at eight rows 7.2 -> 8.2 us, of 896 9.3 -> 8.3)
    const bool pays = p.M <= 8 ? groups >= (p.M > 4 && p.n_jobs > 2 ? 7 : 5) || (groups >= 3 && codes >= (p.M <= 4 ? 3500000 : 10000000)) : groups >= 9 && codes >= 10000000;
    const bool dec = p.M <= 16 && pays && decodes(q) && on_integers(q);
    // Batch kernel at 17 / 64 rows: 2048 x 384 6.3 -> 7.0 / 6.5 -> 7.3, 14336 x 384 8.0 -> 7.4 / 8.2 -> 7.8, 4096 x 640 7.9 -> 7.8 / 8.0 -> 8.2, 896 x 896
    // 8.7 -> 8.3 / 9.0 -> 8.6, 65536 x 128 12.6 -> 10.6 / 12.7 -> 11.5.  Above 64 rows the exchange of shared tiles takes its share: at 128 rows 0.5
    // million codes 9.7 -> 13.2 us, 9 million 12.3 -> 10.5, 17 million 23.2 -> 15.8, 78 million 43.3 -> 45.3.
    // Several matrices at 17 / 64 rows: q|k|v of 896 channels 10.1 -> 10.5 / 11.1 -> 11.4, of 1152 11.9 -> 11.0 / 13.1 -> 11.5 us.
    const bool bat = p.M > 16 && (codes >= 5000000 ? p.M <= 64 || codes <= 40000000 : p.M <= 64 && groups >= (p.n_jobs > 1 ? 9 : 7)) &&
                     (p.dt != UNIQL_BF16 || opt(kOptPrefillConvert) != 1) && batch_supported(q);
    if (small && (dec || bat)) {
      if (!cfg.workspace) {
        int rc = lib_workspace(&cfg.workspace, &cfg.ws_bytes, cfg.stream);
        if (rc != UNIQL_OK) return rc;
      }
      const bool copy_x = p.dt == UNIQL_BF16 && !p.x_f16;
      const size_t own = dec ? decode_workspace_bytes(p.M, p.K + kGroup, n_total) : batch_workspace_bytes(p.M, copy_x ? p.k_in : 0);
      if (cfg.ws_bytes >= at[p.n_jobs] + own + 256) {
        LaunchCfg dc = cfg;
        dc.ws_bytes = (cfg.ws_bytes - at[p.n_jobs]) & ~(size_t)255;
        for (int j = 0; j < p.n_jobs; ++j) {
          __half* o = reinterpret_cast<__half*>(reinterpret_cast<unsigned char*>(cfg.workspace) + dc.ws_bytes + at[j]);
          int rc = launch_pad_scales(p.job[j].scales, p.job[j].zeros, rows[j], G, q.sz_pitch, o, !dec, cfg.stream);
          if (rc != UNIQL_OK) return rc;
          q.job[j].scales = o;
          q.job[j].zeros = o + (size_t)rows[j] * q.sz_pitch;
        }
        if (!dec) return launch_batch(q, dc);
        const int rc = launch_decode(q, dc);
        if (rc != UNIQL_ERR_WORKSPACE && rc != UNIQL_ERR_UNSUPPORTED) return rc;      // (those: nothing was launched)
      }
    }
  }
  // Nine to sixteen rows in bf16: the batch kernel, whose fp16 operands that type had at these sizes before the decode kernel
  // took it (Mamba2-2.7B mixer at 12 rows 28.9 -> 22.0 us).  fp16 stays on exact codes.
  // fp16: its instance that multiplies the codes themselves, by the rule of exact_batch().
  const bool batch = path == UNIQL_PATH_AUTO &&
                     (p.dt == UNIQL_BF16 ? p.M > 8 && p.M <= 16 && batch_supported(p) &&
                                               (!cfg.workspace || cfg.ws_bytes >= batch_workspace_min(true, p.M, p.k_in))
                                         : exact_batch(p));
  if (path == UNIQL_PATH_AUTO)
    path = batch ? UNIQL_PATH_PREFILL : gv ? UNIQL_PATH_GEMV : dec_ok ? UNIQL_PATH_DECODE : (pre_ok ? UNIQL_PATH_PREFILL : UNIQL_PATH_GENERIC);
  if (path == UNIQL_PATH_GEMV) {
    if (!gemv_supported(p)) return UNIQL_ERR_UNSUPPORTED;
    if (!cfg.workspace) {
      int rc = lib_workspace(&cfg.workspace, &cfg.ws_bytes, cfg.stream);
      if (rc != UNIQL_OK) return rc;
    }
    return launch_gemv(p, cfg);
  }
  if (path == UNIQL_PATH_DECODE) {
    if (!decodes(p)) return UNIQL_ERR_UNSUPPORTED;
    if (!cfg.workspace) {
      int rc = lib_workspace(&cfg.workspace, &cfg.ws_bytes, cfg.stream);
      if (rc != UNIQL_OK) return rc;
    }
    // Batches of 9..16: the staged activations of 16 rows do not fit beside the stage ring, which would
    // force the input channels to be split over two groups of blocks and every tile through a hand-over.
    // The integer path streams the activations through the ring instead (one launch, the weights read once);
    // elsewhere two launches over half the batch each re-read the weights but still run more than twice as fast
    // as the split channels (option "decode_split_batch": 2 as described, 1 always two launches, 0 always one
    // launch with staged activations).
    const int sb = opt(kOptDecodeSplitBatch);
    const bool split_batch = sb == 1 || (sb == 2 && !decode_streams_batch(p));
    if (p.M > 8 && split_batch) {
      const int m1 = (p.M + 1) / 2;
      const size_t esz = 2;                               // fp16 / bf16
      Params a = p, b = p;
      a.M = m1;
      b.M = p.M - m1;
      b.x = reinterpret_cast<const unsigned char*>(p.x) + (size_t)m1 * p.ldx * esz;
      b.pos = p.pos ? p.pos + m1 : nullptr;
      for (int j = 0; j < p.n_jobs; ++j)
        b.job[j].y = reinterpret_cast<unsigned char*>(p.job[j].y) + (size_t)m1 * p.job[j].ldy * esz;
      int rc = launch_decode(a, cfg);
      if (rc != UNIQL_OK) return rc;
      return launch_decode(b, cfg);
    }
    return launch_decode(p, cfg);
  }
  if (path == UNIQL_PATH_PREFILL) {
    if (!on_tensor_cores(p)) return UNIQL_ERR_UNSUPPORTED;
    if (!cfg.workspace) {      // only the status word of the workspace is used
      int rc = lib_workspace(&cfg.workspace, &cfg.ws_bytes, cfg.stream);
      if (rc != UNIQL_OK) return rc;
    }
    return launch_prefill(p, cfg);
  }
  return launch_generic(p, cfg);
}

// bf16 at decode sizes ran on the tensor-core kernel until the decode kernel took that type (Qwen2.5-7B layer at two
// rows: 146 us), and it still does where the caller's workspace holds that kernel's scratch but not the decode kernel's.
int dispatch(const Params& p, void* workspace, size_t ws_bytes, void* stream, int path = g_path.load()) {
  if (cudaPeekAtLastError() != cudaSuccess) return UNIQL_ERR_CUDA;
  const int rc = dispatch_as(p, path, workspace, ws_bytes, stream);
  if (rc == UNIQL_ERR_WORKSPACE && path == UNIQL_PATH_AUTO && p.dt != UNIQL_F16 && p.M <= 16)
    return dispatch_as(p, UNIQL_PATH_PREFILL, workspace, ws_bytes, stream);
  return rc;
}

}  // namespace

int uniql::opt(int id) { return g_opt[id].load(std::memory_order_relaxed); }

extern "C" int uniql_set_option(const char* name, int value) {
  if (!name) return UNIQL_ERR_NULL;
  for (int i = 0; i < kOptCount; ++i)
    if (strcmp(name, kOpts[i].name) == 0) { g_opt[i].store(value); return UNIQL_OK; }
  return UNIQL_ERR_SHAPE;
}

extern "C" int uniql_version(void) { return 100; }

extern "C" const char* uniql_status_string(int s) {
  switch (s) {
    case UNIQL_OK: return "ok";
    case UNIQL_ERR_NULL: return "null pointer";
    case UNIQL_ERR_SHAPE: return "bad shape";
    case UNIQL_ERR_ALIGN: return "bad alignment";
    case UNIQL_ERR_DTYPE: return "bad dtype";
    case UNIQL_ERR_UNSUPPORTED: return "unsupported on the forced path";
    case UNIQL_ERR_WORKSPACE: return "workspace too small";
    case UNIQL_ERR_TIMEOUT: return "device-side wait timed out";
    case UNIQL_ERR_CUDA: return "CUDA error";
    default: return "unknown status";
  }
}

extern "C" int uniql_set_path(int path) {
  if (path < UNIQL_PATH_AUTO || path > UNIQL_PATH_GEMV) return UNIQL_ERR_SHAPE;
  g_path.store(path);
  return UNIQL_OK;
}

extern "C" size_t uniql_workspace_bytes(int M, int K, int N_total) {
  if (M < 1 || K < 1 || N_total < 1) return 0;
  // (+ room for the activations re-laid on 8-channel boundaries, see dispatch())
  const size_t relay = (((size_t)M * (size_t)(K + 8) * 2) + 255) / 256 * 256 + 512;
  const int G = (K + kGroup - 1) / kGroup;
  // (an odd number of groups: the copy of the scales and zero-points, see dispatch_as())
  const size_t pad = G % 2 != 0 ? (size_t)N_total * ((G + 7) / 8 * 8) * 4 + 256 * (kMaxJobs + 1) : 0;
  if (M > 16) return prefill_workspace_bytes(M, K) + relay + (M <= 128 ? pad : 0);
  const size_t a = (pad ? decode_workspace_bytes(M, K + kGroup, N_total) : decode_workspace_bytes(M, K, N_total)) + pad;
  const size_t b = M <= 4 ? gemv_workspace_bytes(M, K, N_total) : M > 8 ? batch_workspace_bytes(M, K) : 0;
  return (a > b ? a : b) + relay;
}

extern "C" int uniql_workspace_init(void* workspace, size_t bytes, void* stream) {
  if (!workspace) return UNIQL_ERR_NULL;
  if (((uintptr_t)workspace) & 255) return UNIQL_ERR_ALIGN;
  if (bytes == 0) return UNIQL_ERR_WORKSPACE;
  return cudaMemsetAsync(workspace, 0, bytes, (cudaStream_t)stream) == cudaSuccess ? UNIQL_OK : UNIQL_ERR_CUDA;
}

extern "C" int uniql_workspace_status(void* workspace, int* status) {
  if (!status) return UNIQL_ERR_NULL;
  if (!workspace) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return UNIQL_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_ws_mutex);
    workspace = g_ws[dev];
    if (!workspace) { *status = UNIQL_OK; return UNIQL_OK; }   // never used: nothing can have failed
  }
  int v = 0;
  if (cudaMemcpy(&v, reinterpret_cast<unsigned char*>(workspace) + decode_status_offset(), sizeof(int),
                 cudaMemcpyDeviceToHost) != cudaSuccess)
    return UNIQL_ERR_CUDA;
  *status = v;
  return UNIQL_OK;
}

extern "C" int uniql_qlinear_multi(const void* x, int ldx, int dt, int M, int K, const uniql_chanmap* in_map,
                                   int k_in, int n_jobs, const uniql_job* jobs, void* workspace,
                                   size_t ws_bytes, void* stream) {
  int rc = check_common(x, ldx, dt, M, K);
  if (rc) return rc;
  if (!jobs) return UNIQL_ERR_NULL;
  if (n_jobs < 1 || n_jobs > kMaxJobs) return UNIQL_ERR_SHAPE;
  if (workspace && (((uintptr_t)workspace) & 255)) return UNIQL_ERR_ALIGN;
  Params p;
  memset(&p, 0, sizeof(p));
  rc = compile_map(in_map, k_in, K, &p.imap);
  if (rc) return rc;
  p.x = x; p.ldx = ldx; p.dt = dt; p.M = M; p.K = K; p.k_in = p.imap.total;
  if (ldx < p.k_in) return UNIQL_ERR_SHAPE;
  p.n_jobs = n_jobs;
  for (int j = 0; j < n_jobs; ++j) {
    const uniql_job& s = jobs[j];
    rc = check_weight(s.packed_w, s.scales, s.zeros, s.N);
    if (rc) return rc;
    if (!s.y) return UNIQL_ERR_NULL;
    if ((((uintptr_t)s.y) & 1) || (s.bias && (((uintptr_t)s.bias) & 1))) return UNIQL_ERR_ALIGN;
    JobDev& d = p.job[j];
    rc = compile_map(s.out_map, s.k_out, s.N, &d.omap);
    if (rc) return rc;
    d.w = s.packed_w; d.scales = (const __half*)s.scales; d.zeros = (const __half*)s.zeros;
    d.bias = s.bias; d.y = s.y; d.ldy = s.ldy; d.N = s.N; d.k_out = d.omap.total;
    if (s.ldy < d.k_out) return UNIQL_ERR_SHAPE;
  }
  return dispatch(p, workspace, ws_bytes, stream);
}

extern "C" int uniql_qlinear_ex(const void* x, int ldx, int dt, const uint8_t* packed_w, const void* scales,
                                const void* zeros, const void* bias, int M, int K, int N,
                                const uniql_chanmap* in_map, int k_in, const uniql_chanmap* out_map,
                                int k_out, void* y, int ldy, void* workspace, size_t ws_bytes, void* stream) {
  uniql_job job;
  memset(&job, 0, sizeof(job));
  job.packed_w = packed_w; job.scales = scales; job.zeros = zeros; job.bias = bias;
  job.N = N; job.k_out = k_out; job.out_map = out_map; job.y = y; job.ldy = ldy;
  return uniql_qlinear_multi(x, ldx, dt, M, K, in_map, k_in, 1, &job, workspace, ws_bytes, stream);
}

extern "C" int uniql_qlinear(const void* x, const uint8_t* packed_w, const void* scales, const void* zeros,
                             int M, int K, int N, int k_in, int k_out, void* y, void* stream) {
  return uniql_qlinear_ex(x, k_in, UNIQL_F16, packed_w, scales, zeros, nullptr, M, K, N, nullptr, k_in,
                          nullptr, k_out, y, k_out, nullptr, 0, stream);
}

namespace {

// Rotation frequencies as fractions of a turn.  A model calls with the same head_dim and theta (or table) for every
// layer and token, and 64 powers and extended-precision fractions cost 7 us of host time, three times the launch: each
// thread keeps the table it made last, next to the arguments it was made from.
void rope_turns(int head_dim, double theta, const double* inv_freq, unsigned long long* turn) {
  struct Table { int head_dim = 0; bool given = false; double theta = 0, freq[kMaxHalfDim]; unsigned long long turn[kMaxHalfDim]; };
  static thread_local Table t;
  const int half = head_dim / 2;
  const bool same = t.head_dim == head_dim && t.given == (inv_freq != nullptr) &&
                    (inv_freq ? memcmp(t.freq, inv_freq, (size_t)half * sizeof(double)) == 0 : t.theta == theta);
  if (!same) {
    t.head_dim = head_dim; t.given = inv_freq != nullptr; t.theta = theta;
    if (inv_freq) memcpy(t.freq, inv_freq, (size_t)half * sizeof(double));
    for (int i = 0; i < half; ++i)
      t.turn[i] = rope_turn_of(inv_freq ? inv_freq[i] : pow(theta, -2.0 * (double)i / (double)head_dim));
  }
  memcpy(turn, t.turn, (size_t)half * sizeof(turn[0]));
}

// Q and K projections with the rotary epilogue and, when wv is given, the V projection (plain rows, the
// leading v_keep of every key-value head) as a third job of the same launch.
int qkv_rope_impl(const void* x, int ldx, int dt, const uint8_t* wq, const void* sq, const void* zq,
                  const uint8_t* wk, const void* sk, const void* zk, const uint8_t* wv, const void* sv,
                  const void* zv, const void* bq, const void* bk, const void* bv, int M, int K, int n_q_heads,
                  int n_kv_heads, int head_dim, int head_keep, int v_keep, const int32_t* retained_idx,
                  const int32_t* pos, double theta, const double* inv_freq, void* q_out, int ldq, void* k_out,
                  int ldk, void* v_out, int ldv, void* workspace, size_t ws_bytes, void* stream) {
  int rc = check_common(x, ldx, dt, M, K);
  if (rc) return rc;
  if (!retained_idx || !pos || !q_out || !k_out) return UNIQL_ERR_NULL;
  if (n_q_heads < 1 || n_kv_heads < 1 || (n_q_heads % n_kv_heads) != 0) return UNIQL_ERR_SHAPE;
  if (head_dim < 2 || (head_dim & 1) || head_dim > 2 * kMaxHalfDim) return UNIQL_ERR_SHAPE;
  if (head_keep < 2 || (head_keep & 1) || head_keep > head_dim) return UNIQL_ERR_SHAPE;
  if (!inv_freq && !(theta > 0.0)) return UNIQL_ERR_SHAPE;
  if (ldx < K) return UNIQL_ERR_SHAPE;   // the hidden dimension D_h is never pruned (Section 3.4)
  if (ldq < n_q_heads * head_keep || ldk < n_kv_heads * head_keep) return UNIQL_ERR_SHAPE;
  if ((((uintptr_t)q_out) & 1) || (((uintptr_t)k_out) & 1) || (((uintptr_t)retained_idx) & 3) ||
      (((uintptr_t)pos) & 3))
    return UNIQL_ERR_ALIGN;
  if ((bq && (((uintptr_t)bq) & 1)) || (bk && (((uintptr_t)bk) & 1))) return UNIQL_ERR_ALIGN;
  if (workspace && (((uintptr_t)workspace) & 255)) return UNIQL_ERR_ALIGN;
  rc = check_weight(wq, sq, zq, n_q_heads * head_dim);
  if (rc) return rc;
  rc = check_weight(wk, sk, zk, n_kv_heads * head_dim);
  if (rc) return rc;
  if (wv) {
    if (!v_out) return UNIQL_ERR_NULL;
    if (v_keep < 1 || v_keep > head_dim || ldv < n_kv_heads * v_keep) return UNIQL_ERR_SHAPE;
    if ((((uintptr_t)v_out) & 1) || (bv && (((uintptr_t)bv) & 1))) return UNIQL_ERR_ALIGN;
    rc = check_weight(wv, sv, zv, n_kv_heads * head_dim);
    if (rc) return rc;
  }

  Params p;
  memset(&p, 0, sizeof(p));
  compile_map(nullptr, K, K, &p.imap);
  p.x = x; p.ldx = ldx; p.dt = dt; p.M = M; p.K = K; p.k_in = K;
  p.n_jobs = wv ? 3 : 2;
  p.idx = retained_idx; p.pos = pos;
  rope_turns(head_dim, theta, inv_freq, p.rope_turn);
  for (int j = 0; j < 2; ++j) {
    JobDev& d = p.job[j];
    int nh = j == 0 ? n_q_heads : n_kv_heads;
    d.w = j == 0 ? wq : wk;
    d.scales = (const __half*)(j == 0 ? sq : sk);
    d.zeros = (const __half*)(j == 0 ? zq : zk);
    d.bias = j == 0 ? bq : bk;
    d.y = j == 0 ? q_out : k_out;
    d.ldy = j == 0 ? ldq : ldk;
    d.N = nh * head_dim;
    d.k_out = nh * head_keep;
    uniql_chanmap hm;
    hm.n_fam = 1;
    hm.fam[0] = uniql_family{0, head_dim / 2, head_keep / 2, 2 * nh};
    compile_map(&hm, 0, d.N, &d.omap);
    d.rope = RopeDesc{1, nh, j == 0 ? n_q_heads / n_kv_heads : 1, head_dim, head_keep};
  }
  if (wv) {
    JobDev& d = p.job[2];
    d.w = wv; d.scales = (const __half*)sv; d.zeros = (const __half*)zv; d.bias = bv;
    d.y = v_out; d.ldy = ldv; d.N = n_kv_heads * head_dim;
    uniql_chanmap hm;
    hm.n_fam = 1;
    hm.fam[0] = uniql_family{0, head_dim, v_keep, n_kv_heads};
    rc = compile_map(&hm, 0, d.N, &d.omap);
    if (rc) return rc;
    d.k_out = d.omap.total;
  }
  return dispatch(p, workspace, ws_bytes, stream);
}

}  // namespace

extern "C" int uniql_qk_rope_proj(const void* x, int ldx, int dt, const uint8_t* wq, const void* sq,
                                  const void* zq, const uint8_t* wk, const void* sk, const void* zk,
                                  const void* bq, const void* bk, int M, int K, int n_q_heads,
                                  int n_kv_heads, int head_dim, int head_keep, const int32_t* retained_idx,
                                  const int32_t* pos, double theta, const double* inv_freq, void* q_out,
                                  int ldq, void* k_out, int ldk, void* workspace, size_t ws_bytes,
                                  void* stream) {
  return qkv_rope_impl(x, ldx, dt, wq, sq, zq, wk, sk, zk, nullptr, nullptr, nullptr, bq, bk, nullptr, M, K,
                       n_q_heads, n_kv_heads, head_dim, head_keep, 0, retained_idx, pos, theta, inv_freq, q_out,
                       ldq, k_out, ldk, nullptr, 0, workspace, ws_bytes, stream);
}

extern "C" int uniql_qkv_rope_proj(const void* x, int ldx, int dt, const uint8_t* wq, const void* sq,
                                   const void* zq, const uint8_t* wk, const void* sk, const void* zk,
                                   const uint8_t* wv, const void* sv, const void* zv, const void* bq,
                                   const void* bk, const void* bv, int M, int K, int n_q_heads, int n_kv_heads,
                                   int head_dim, int head_keep, int v_keep, const int32_t* retained_idx,
                                   const int32_t* pos, double theta, const double* inv_freq, void* q_out,
                                   int ldq, void* k_out, int ldk, void* v_out, int ldv, void* workspace,
                                   size_t ws_bytes, void* stream) {
  if (!wv) return UNIQL_ERR_NULL;
  return qkv_rope_impl(x, ldx, dt, wq, sq, zq, wk, sk, zk, wv, sv, zv, bq, bk, bv, M, K, n_q_heads, n_kv_heads,
                       head_dim, head_keep, v_keep, retained_idx, pos, theta, inv_freq, q_out, ldq, k_out, ldk,
                       v_out, ldv, workspace, ws_bytes, stream);
}

namespace {

// SwiGLU MLP on the tensor-core kernel, two launches.  The first takes gate and up as a pair (their retained
// rows interleaved in every tile) and writes h = silu(x Wg^T) * (x Wu^T); the second is the plain down
// projection over the leading k_int channels of h.
int mlp_tensor_core(const void* x, int ldx, int dt, const uint8_t* wg, const void* sg, const void* zg, const uint8_t* wu,
                    const void* su, const void* zu, const uint8_t* wd, const void* sd, const void* zd, int M, int hidden,
                    int inter, int k_int, void* h, int ldh, void* y, int ldy, const LaunchCfg& cfg_in) {
  if ((hidden % kGroup) != 0 || (inter % kGroup) != 0) return UNIQL_ERR_SHAPE;
  Params a;
  memset(&a, 0, sizeof(a));
  compile_map(nullptr, hidden, hidden, &a.imap);
  a.x = x; a.ldx = ldx; a.dt = dt; a.M = M; a.K = hidden; a.k_in = hidden;
  a.n_jobs = 2;
  for (int j = 0; j < 2; ++j) {
    JobDev& jd = a.job[j];
    compile_map(nullptr, k_int, inter, &jd.omap);
    jd.w = j == 0 ? wg : wu;
    jd.scales = (const __half*)(j == 0 ? sg : su);
    jd.zeros = (const __half*)(j == 0 ? zg : zu);
    jd.y = h; jd.ldy = ldh; jd.N = inter; jd.k_out = k_int;
    jd.pair = j + 1;
  }
  // bf16 on the batch kernel: the gated launch leaves h as fp16 too, in rows of whole 128-byte lines at the end of the workspace,
  // and the down projection reads that copy: a pass over h in between is a launch of its own (Llama-3-8B layer at 34 rows, with
  // the kept blocks converted on their way, 77.3 -> 72.0 us).  Where there is room beside everything that the two launches may use.
  // Not above 128 rows: there the second store of every output cost the gated launch what the pass takes (Qwen2.5-7B at 2048
  // rows 730 -> 744 us, at 677 336 -> 339 us).
  // (path and option are read here once for both launches: a switch set by another thread in between must not send the down
  //  projection to a copy that was not written, nor the copy to a kernel that takes it for bf16)
  const int ld16 = (k_int + 63) / 64 * 64, path = g_path.load();
  const size_t h16_bytes = ((size_t)M * ld16 * 2 + 255) & ~(size_t)255;
  const bool h16 = dt == UNIQL_BF16 && M > 16 && batch_supported(a) && (path == UNIQL_PATH_AUTO || path == UNIQL_PATH_PREFILL) &&
                   opt(kOptPrefillConvert) != 1 && cfg_in.ws_bytes >= h16_bytes + prefill_workspace_bytes(M, hidden) + 256;
  LaunchCfg cfg = cfg_in;
  if (h16) {
    cfg.ws_bytes = (cfg_in.ws_bytes - h16_bytes) & ~(size_t)255;
    a.job[0].y16 = reinterpret_cast<__half*>(reinterpret_cast<unsigned char*>(cfg_in.workspace) + cfg.ws_bytes);
    a.job[0].ld16 = ld16;
  }
  if (!prefill_supported(a) || (M <= 16 && dt == UNIQL_F16 && !exact_batch(a))) return UNIQL_ERR_UNSUPPORTED;   // (nothing launched)
  int rc = h16 ? launch_batch(a, cfg) : launch_prefill(a, cfg);
  if (rc != UNIQL_OK) return rc;
  Params b;
  memset(&b, 0, sizeof(b));
  compile_map(nullptr, k_int, inter, &b.imap);
  b.x = h; b.ldx = ldh; b.dt = dt; b.M = M; b.K = inter; b.k_in = k_int;
  if (h16) { b.x = a.job[0].y16; b.ldx = ld16; b.x_f16 = 1; }
  b.n_jobs = 1;
  JobDev& jd = b.job[0];
  compile_map(nullptr, hidden, hidden, &jd.omap);
  jd.w = wd; jd.scales = (const __half*)sd; jd.zeros = (const __half*)zd;
  jd.y = y; jd.ldy = ldy; jd.N = hidden; jd.k_out = hidden;
  return dispatch(b, cfg.workspace, cfg.ws_bytes, cfg.stream, path);
}

}  // namespace

extern "C" size_t uniql_mlp_workspace_bytes(int M, int hidden, int inter) {
  if (M < 1 || hidden < 1 || inter < 1) return 0;
  // (an odd number of groups: the down projection's copy of the scales and zero-points, see dispatch_as())
  const int G = (inter + kGroup - 1) / kGroup;
  const size_t pad = G % 2 != 0 && M <= 128 ? (size_t)hidden * ((G + 7) / 8 * 8) * 4 + 768 : 0;
  // tensor-core kernel, two launches (+ up to 128 rows the fp16 copies of both activations of bf16 at once)
  if (M > 16)
    return prefill_workspace_bytes(M, hidden > inter ? hidden : inter) + pad +
           (M <= 128 ? (size_t)M * (((hidden < inter ? hidden : inter) + 63) / 64 * 64) * 2 + 512 : 0);
  // (16 rows or fewer in bf16 also run on the tensor-core kernel: room for its fp16 copy of the activations)
  const size_t a = mlp_decode_workspace_bytes(M, hidden, inter), b = prefill_workspace_bytes(M, hidden > inter ? hidden : inter);
  size_t c = 0;
  if (M <= 4) {
    const size_t c0 = gemv_workspace_bytes(M, hidden, 2 * inter), c1 = gemv_workspace_bytes(M, inter, hidden);
    c = c0 > c1 ? c0 : c1;
  }
  if (pad) {
    const size_t down = decode_workspace_bytes(M, inter + kGroup, hidden) + pad;
    c = c > down ? c : down;
  }
  return a > b ? (a > c ? a : c) : (b > c ? b : c);
}

namespace {

// The SwiGLU block for either activation type: decode sizes on the decode kernel, the rest on the tensor cores.
int mlp_block(const void* x, int ldx, int dt, const uint8_t* wg, const void* sg, const void* zg, const uint8_t* wu,
              const void* su, const void* zu, const uint8_t* wd, const void* sd, const void* zd, int M, int hidden,
              int inter, int k_int, void* h, int ldh, void* y, int ldy, int fuse, void* workspace, size_t ws_bytes,
              void* stream) {
  if (!x || !h || !y) return UNIQL_ERR_NULL;
  if (M < 1 || hidden < kGroup || inter < kGroup || k_int < 1 || k_int > inter) return UNIQL_ERR_SHAPE;
  if (ldx < hidden || ldh < k_int || ldy < hidden) return UNIQL_ERR_SHAPE;
  if (fuse < -1 || fuse > 1) return UNIQL_ERR_SHAPE;
  int rc = check_weight(wg, sg, zg, inter);
  if (!rc) rc = check_weight(wu, su, zu, inter);
  if (!rc) rc = check_weight(wd, sd, zd, hidden);
  if (rc) return rc;
  if ((((uintptr_t)x) | ((uintptr_t)h) | ((uintptr_t)y)) & 1) return UNIQL_ERR_ALIGN;
  if (workspace && (((uintptr_t)workspace) & 255)) return UNIQL_ERR_ALIGN;
  if (cudaPeekAtLastError() != cudaSuccess) return UNIQL_ERR_CUDA;
  LaunchCfg cfg{workspace, ws_bytes, (cudaStream_t)stream};
  if (!cfg.workspace) {
    rc = lib_workspace(&cfg.workspace, &cfg.ws_bytes, cfg.stream);
    if (rc != UNIQL_OK) return rc;
  }
  auto tensor_core = [&]() -> int {
    return mlp_tensor_core(x, ldx, dt, wg, sg, zg, wu, su, zu, wd, sd, zd, M, hidden, inter, k_int, h, ldh, y, ldy, cfg);
  };
  if (M > 16) return fuse == 1 ? UNIQL_ERR_UNSUPPORTED : tensor_core();
  MlpDecode d;
  memset(&d, 0, sizeof(d));
  d.dt = dt;
  d.x = x; d.ldx = ldx; d.M = M; d.hidden = hidden; d.inter = inter; d.k_int = k_int;
  d.wg = wg; d.wu = wu; d.wd = wd;
  d.sg = (const __half*)sg; d.zg = (const __half*)zg; d.su = (const __half*)su; d.zu = (const __half*)zu;
  d.sd = (const __half*)sd; d.zd = (const __half*)zd;
  d.h = h; d.ldh = ldh; d.y = y; d.ldy = ldy;
  d.decode_only = g_path.load() == UNIQL_PATH_DECODE;
  if (dt != UNIQL_F16) {
    // bf16: the decode kernel where its rules and the workspace allow it, else the tensor cores as for larger batches
    const bool too_small = workspace && ws_bytes < mlp_decode_workspace_bytes(M, hidden, inter);
    if ((g_path.load() != UNIQL_PATH_AUTO && g_path.load() != UNIQL_PATH_DECODE) || too_small || !mlp_decode_supported(d))
      return tensor_core();
  }
  // the batch kernel on exact codes, both products (a decode launch behind a batch launch cannot come in beside it)
  if (dt == UNIQL_F16 && M > 8 && fuse != 1 && g_path.load() == UNIQL_PATH_AUTO && mlp_decode_supported(d)) {
    rc = tensor_core();
    if (rc != UNIQL_ERR_UNSUPPORTED) return rc;
  }
  // one to four rows: two launches of the streaming kernel (unless one launch or the persistent kernel is asked for)
  if (fuse != 1 && gemv_mlp_supported(d) &&
      (g_path.load() == UNIQL_PATH_GEMV ||
       (g_path.load() == UNIQL_PATH_AUTO && (opt(kOptGemvFirst) == 1 || !mlp_decode_supported(d)))))
    return launch_gemv_mlp(d, cfg);
  if (g_path.load() == UNIQL_PATH_GEMV) return UNIQL_ERR_UNSUPPORTED;
  if (!mlp_decode_supported(d)) return UNIQL_ERR_UNSUPPORTED;
  auto run = [&](const MlpDecode& q) -> int {
    // fuse = -1 takes two launches: on B200 the launch boundary (programmatic dependent launch) costs less
    // than the grid-wide barrier of the single launch (measured 29.2 us against 32.6 us per Llama-3-8B layer)
    return launch_mlp_decode(q, fuse == 1 ? 1 : 0, cfg);
  };
  // (nine to sixteen rows: one pass with streamed activations, or under option "decode_split_batch" 0 / 1 as for
  // the plain decode path)
  if (M > 8 && fuse != 1 && !(opt(kOptDecodeSplitBatch) == 2 && opt(kOptDecodeXstream) != 0 && opt(kOptDecodeI8) != 0)) {
    const int m1 = (M + 1) / 2;
    MlpDecode a = d, b = d;
    a.M = m1;
    b.M = M - m1;
    b.x = reinterpret_cast<const unsigned char*>(x) + (size_t)m1 * ldx * 2;
    b.h = reinterpret_cast<unsigned char*>(h) + (size_t)m1 * ldh * 2;
    b.y = reinterpret_cast<unsigned char*>(y) + (size_t)m1 * ldy * 2;
    if (!mlp_decode_supported(b)) return UNIQL_ERR_UNSUPPORTED;
    rc = run(a);
    return rc ? rc : run(b);
  }
  return run(d);
}

}  // namespace

extern "C" int uniql_mlp_swiglu_decode(const void* x, int ldx, const uint8_t* wg, const void* sg, const void* zg,
                                       const uint8_t* wu, const void* su, const void* zu, const uint8_t* wd,
                                       const void* sd, const void* zd, int M, int hidden, int inter, int k_int,
                                       void* h, int ldh, void* y, int ldy, int fuse, void* workspace,
                                       size_t ws_bytes, void* stream) {
  return mlp_block(x, ldx, UNIQL_F16, wg, sg, zg, wu, su, zu, wd, sd, zd, M, hidden, inter, k_int, h, ldh, y, ldy, fuse,
                   workspace, ws_bytes, stream);
}

extern "C" int uniql_mlp_swiglu(const void* x, int ldx, int dt, const uint8_t* wg, const void* sg, const void* zg,
                                const uint8_t* wu, const void* su, const void* zu, const uint8_t* wd, const void* sd,
                                const void* zd, int M, int hidden, int inter, int k_int, void* h, int ldh, void* y,
                                int ldy, void* workspace, size_t ws_bytes, void* stream) {
  if (dt != UNIQL_F16 && dt != UNIQL_BF16) return UNIQL_ERR_DTYPE;
  return mlp_block(x, ldx, dt, wg, sg, zg, wu, su, zu, wd, sd, zd, M, hidden, inter, k_int, h, ldh, y, ldy, -1, workspace,
                   ws_bytes, stream);
}
