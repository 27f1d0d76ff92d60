// unet_api.cu -- the warm-start U-Net runtime behind include/lbnci_unet.h: layer table,
// activation and gradient buffers, the forward and backward launch sequences, Adam.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "lbnci_unet.h"
#include "unet_kernels.cuh"
#include "unet_conv.cuh"
#include "lb_launch.h"

// Error word of the single tensor-core convolutions (lbu_conv3x3, lbu_conv3x3_wgrad): bit 0 set
// when a bounded mbarrier wait expired (the launch then wrote no output). A network's kernels
// set a word of its own (lbu_net::tc_err).
__device__ int g_tc_err;
static std::atomic<bool> g_single_used{false};  // some single call has run such a kernel

using lbu::bf16;

namespace {

constexpr int kInPad = 32;  // input channels are padded to one K chunk of the convolution

struct LayerHost {
  int cout, cin, cin_pad, taps;
  long long w_off, b_off, wb_off, wt_off;
};

bool valid_config(const lbu_config* c, std::string* why) {
  if (!c) return *why = "null config", false;
  if (c->levels < 2 || c->levels > 6) return *why = "levels must be 2..6", false;
  if (c->base <= 0 || c->base % 32 != 0) return *why = "base must be a positive multiple of 32", false;
  if (c->base * (1 << (c->levels - 1)) > 1024) return *why = "widest level exceeds 1024 channels", false;
  if (c->in_ch < 1 || c->in_ch > kInPad) return *why = "in_ch must be 1..32", false;
  if (c->out_ch < 1 || c->out_ch > lbu::kMaxOut) return *why = "out_ch must be 1..8", false;
  if (c->base > lbu::kMaxHeadIn) return *why = "base exceeds the head kernel's 256 input channels", false;
  const int f = 1 << (c->levels - 1);
  if (c->H <= 0 || c->W <= 0 || c->H % f || c->W % f) return *why = "H and W must be multiples of 2^(levels-1)", false;
  if (c->max_batch <= 0) return *why = "max_batch must be positive", false;
  if ((long long)c->max_batch * c->H * c->W > (1LL << 30) / 64) return *why = "max_batch * H * W too large", false;
  return true;
}

std::vector<LayerHost> layer_table(const lbu_config* c) {
  std::vector<LayerHost> L;
  auto add = [&](int cout, int cin, int taps) {
    LayerHost l{};
    l.cout = cout;
    l.cin = cin;
    l.cin_pad = taps == 9 ? ((cin + 31) / 32) * 32 : cin;
    l.taps = taps;
    L.push_back(l);
  };
  std::vector<int> C(c->levels);
  for (int l = 0; l < c->levels; ++l) C[l] = c->base << l;
  int cin = c->in_ch;
  for (int l = 0; l < c->levels; ++l) {
    add(C[l], cin, 9);
    add(C[l], C[l], 9);
    cin = C[l];
  }
  for (int l = c->levels - 2; l >= 0; --l) {
    add(C[l], C[l + 1], 9);
    add(C[l], 2 * C[l], 9);
    add(C[l], C[l], 9);
  }
  add(c->out_ch, C[0], 1);
  long long off = 0, wb = 0, wt = 0;
  for (size_t i = 0; i < L.size(); ++i) {
    LayerHost& l = L[i];
    l.w_off = off;
    off += (long long)l.cout * l.taps * l.cin;
    l.b_off = off;
    off += l.cout;
    l.wb_off = wb;
    wb += (long long)l.cout * l.taps * l.cin_pad;
    if (l.taps == 9 && i > 0) {  // the first layer needs no data gradient
      l.wt_off = wt;
      wt += (long long)l.cout * 9 * l.cin_pad;
    } else {
      l.wt_off = -1;
    }
  }
  return L;
}

long long total_params(const std::vector<LayerHost>& L) {
  const LayerHost& b = L.back();
  return b.b_off + b.cout;
}

// wgrad partition: splits of the pixel range so that the grid has about 4 waves of blocks
struct WgradPlan {
  int BM, BN, nsplit, pps;
};
WgradPlan wgrad_plan(int P, int cin, int cout) {
  WgradPlan w;
  w.BM = cout % 64 == 0 ? 64 : 32;
  w.BN = cin % 64 == 0 ? 64 : 32;
  const int blocks_xy = (cout / w.BM) * 9 * (cin / w.BN);
  int ns = (4 * 152 + blocks_xy - 1) / blocks_xy;
  ns = std::max(1, std::min(ns, (P + 255) / 256));
  int pps = (P + ns - 1) / ns;
  pps = (pps + 31) / 32 * 32;
  w.pps = pps;
  w.nsplit = (P + pps - 1) / pps;
  return w;
}
size_t wgrad_bytes(const WgradPlan& w, int cin, int cout) {
  return ((size_t)w.nsplit * cout * 9 * cin + (size_t)w.nsplit * cout) * sizeof(float);
}

constexpr int kSmemMax = 227 * 1024, kSmemSm = 228 * 1024;

// Partition of the tensor-memory weight gradient (conv3x3_wgrad_tma_kernel) over B images of
// H x W positions (the low-resolution input's when up): tiles of eight rows x 32 columns
// (four rows when up, whose stage holds four tiles of dy), as many stages as the shared
// memory of one or two CTAs holds, and as many splits as fill the 152 multiprocessors once.
struct WgradTmaPlan {
  bool ok = false;
  int BN, rowb, smem;
  lbu::WgradTma a;
};
WgradTmaPlan wgrad_tma_plan(int B, int H, int W, int cin, int cout, int up) {
  WgradTmaPlan p;
  if (cin % 32 || cout % 32) return p;
  p.rowb = cin % 64 == 0 ? 128 : 64;
  p.BN = cout % 64 == 0 ? 64 : 32;
  if (up && p.rowb != 128) return p;
  lbu::WgradTma& a = p.a;
  a = lbu::WgradTma{};
  a.H = H;
  a.W = W;
  a.up = up;
  a.TW = W >= 32 ? 32 : 16;
  a.TH = std::min(H, up ? 4 : 8);
  a.pitch = a.TW + 2;
  a.tiles_x = (W + a.TW - 1) / a.TW;
  a.tiles_y = (H + a.TH - 1) / a.TH;
  a.ntile = B * a.tiles_x * a.tiles_y;
  a.Cin = cin;
  a.Cout = cout;
  const int npar = up ? 4 : 1, nacc = up ? 8 : (p.rowb == 64 ? 3 : 5);
  a.x_bytes = (((a.TH + 2) * a.pitch + 1) * p.rowb + 1023) / 1024 * 1024;
  a.d_bytes = (a.TH * a.TW * p.BN * 2 + 1023) / 1024 * 1024;
  const int stage = a.x_bytes + npar * a.d_bytes;
  a.cols = 32;
  while (a.cols < nacc * p.BN) a.cols *= 2;
  const int occ = a.cols <= 256 && 2 * (2 * stage + 2048) <= kSmemSm ? 2 : 1;
  a.nstage = std::min(lbu::kWgradMaxStage, (kSmemSm / occ - 3072) / stage);
  if (a.nstage < 2) return p;
  a.tail = std::max(a.nstage * stage, 8192);
  // no more CTAs on a multiprocessor than its tensor memory serves
  p.smem = std::max(a.tail + (int)sizeof(lbu::WgradTail), kSmemSm / (512 / a.cols + 1) - 1024 + 16);
  if (p.smem > kSmemMax) return p;
  const int blocks = (cin / (p.rowb / 2)) * (cout / p.BN);
  a.nsplit = std::max(1, std::min(a.ntile, 152 * occ / blocks));
  p.ok = true;
  return p;
}
size_t wgrad_tma_bytes(const WgradTmaPlan& p) {
  const lbu::WgradTma& a = p.a;
  return p.ok ? ((size_t)a.nsplit * a.Cout * (a.up ? 16 : 9) * a.Cin + (size_t)a.nsplit * a.Cout) * sizeof(float) : 0;
}
// Scratch of a weight gradient by either kernel, with or without upsampled input.
size_t wgrad_work(int B, int H, int W, int cin, int cout) {
  size_t n = wgrad_bytes(wgrad_plan(B * H * W, cin, cout), cin, cout);
  n = std::max(n, wgrad_tma_bytes(wgrad_tma_plan(B, H, W, cin, cout, 0)));
  if (H % 2 == 0 && W % 2 == 0) n = std::max(n, wgrad_tma_bytes(wgrad_tma_plan(B, H / 2, W / 2, cin, cout, 1)));
  return n;
}

thread_local std::string g_err;

// One launch of conv3x3_tma_kernel or, rows, conv3x3_rows_kernel: tensor maps, tile and grid
// of a convolution's operands.
struct ConvPlan {
  bool ok = false, rows = false;
  CUtensorMap mx, mw;
  lbu::ConvTma a;
  lbu::ConvRows r;
  dim3 grid;
  int smem = 0, BN = 0, rowb = 0;
};

// The plans of a network's launches, one per layer and direction, kept for the batch they
// were made for: a layer's operands are the network's own buffers.
struct ConvCache {
  int B = -1;
  ConvPlan p;
};
struct WgradCache {
  int B = -1;
  WgradTmaPlan p;
  lbu::WgradMaps maps;
};

}  // namespace

// What the calls that synchronise read back: the loss, the network's error word and the number
// of parameter updates left out since it was set.
struct Report {
  double loss;
  int err, skipped;
};

struct lbu_net {
  lbu_config cfg;
  std::vector<LayerHost> L;
  long long nparams = 0;
  cudaStream_t stream = nullptr;
  int device = 0;
  float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
  bf16 *wb = nullptr, *wt = nullptr;
  lbu::LayerDev* Ldev = nullptr;
  // activations, per level l (image H>>l x W>>l, width C_l)
  std::vector<bf16*> ea, cat, pool, da, db, gA, gB, gCat, gU, gPool;
  bf16* x0 = nullptr;
  float *y = nullptr, *dy = nullptr, *xstage = nullptr, *ystage = nullptr;
  float* work = nullptr;
  size_t work_bytes = 0;
  double *partial = nullptr, *loss = nullptr;  // loss: a Report
  int* tc_err = nullptr;  // in that Report
  int npartial = 0;
  float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  long long t = 0;
  long long launches = 0;
  std::vector<ConvCache> conv_cache;    // forward of layer i: i, data gradient: layers + i
  std::vector<WgradCache> wgrad_cache;  // layer i
  std::vector<void*> allocs;
  std::string err;
};

namespace {

lb_status fail(lbu_net* n, lb_status st, const std::string& msg) {
  if (n) n->err = msg; else g_err = msg;
  return st;
}
lb_status cuda_fail(lbu_net* n, cudaError_t e, const char* where) {
  (void)cudaGetLastError();
  return fail(n, LB_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}
#define LBU_CUDA(n, call)                                        \
  do {                                                           \
    cudaError_t e_ = (call);                                     \
    if (e_ != cudaSuccess) return cuda_fail((n), e_, #call);     \
  } while (0)

int width(const lbu_net* n, int l) { return n->cfg.base << l; }
int Hl(const lbu_net* n, int l) { return n->cfg.H >> l; }
int Wl(const lbu_net* n, int l) { return n->cfg.W >> l; }

template <typename T>
lb_status dalloc(lbu_net* n, T** p, size_t count) {
  void* q = nullptr;
  cudaError_t e = cudaMalloc(&q, std::max<size_t>(count, 1) * sizeof(T));
  if (e != cudaSuccess) return cuda_fail(n, e, "cudaMalloc");
  n->allocs.push_back(q);
  *p = static_cast<T*>(q);
  return LB_OK;
}

int grid_for(long long work, int threads) {
  long long b = (work + threads - 1) / threads;
  return (int)std::max<long long>(1, std::min<long long>(b, 152LL * 16));
}

// ------------------------------------------------------------------ tensor-core convolution
bool encode_tiled(CUtensorMap* m, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                  const cuuint32_t* box, int rowb) {
  auto fn = lbnci::encode_fn();
  if (!fn) return false;
  const cuuint32_t es[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, rowb == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The tile of a convolution over B images of H x W positions (the low-resolution input's
// when up): among tiles of 16 rows x 8 k columns (every operand row a pixel) and tiles of
// TH rows x min(W, 126) columns (rows of the operand run through the pitched tile), those
// whose operands fit, the one with the smallest estimated time. The estimate counts, per
// multiprocessor, waves of resident CTAs; a wave takes the first copy (about 2,000 cycles),
// the MMAs (32 + N/4 cycles each, the operands' bytes) or the copies (about 50 bytes a
// cycle), whichever is longer, and the drain (30 cycles a column of a group's accumulators,
// 50 with a mask); two CTAs overlap one's drain with the other's MMAs.
bool plan_tile(int B, int H, int W, int cin, int cout, int up, bool mask, ConvPlan* p) {
  p->rowb = cin % 64 == 0 ? 128 : 64;
  const int nchunk = cin / (p->rowb / 2), npar = up ? 4 : 1, ni = 9 * nchunk;
  double best = 1e30;
  auto consider = [&](int BN, int TH, int TW, bool linear) {
    const int bstage = BN * p->rowb;
    const int stages = std::min(std::min(ni, lbu::kConvMaxStage), std::max(3, 36864 / bstage));
    const int pitch = TW + 2, sbo = linear ? 8 : pitch, mstart = linear ? 128 : 8;
    const int nm = linear ? (TH * pitch - 2 + 127) / 128 : TW / 8;
    const int ncols = nm * npar * BN;
    if (ncols > 512 || TW + 2 > 256 || TH + 2 > 256) return;
    int cols = 32;
    while (cols < ncols) cols *= 2;
    // rows of the tile in shared memory: the copy's, and what the last M tile reads beyond it
    const int reach = (nm - 1) * mstart + 15 * sbo + 7 + 2 * pitch + 2 + 1;
    const int rows = std::max((TH + 2) * pitch, reach);
    const int a_stride = (rows * p->rowb + 1023) / 1024 * 1024;
    const int body = std::max(nchunk * a_stride + stages * bstage, 2 * 128 * BN * 2);
    const int tail = (body + 15) / 16 * 16;
    // at most 512/cols CTAs per SM: none ever waits for another's tensor memory
    const int smem = std::max(tail + (int)sizeof(lbu::ConvTail), kSmemSm / (512 / cols + 1) - 1024 + 16);
    if (smem > kSmemMax) return;
    const int occ = std::min(std::min(kSmemSm / (smem + 1024), 512 / cols), 3);
    if (occ < 1) return;
    const int tiles_x = (W + TW - 1) / TW, tiles_y = (H + TH - 1) / TH;
    const double ctas = (double)B * tiles_x * tiles_y * (cout / BN);
    const double waves = std::ceil(ctas / (152.0 * occ));
    const double mma = (double)nm * npar * ni * (p->rowb / 32) * (32 + BN / 4);
    const double copy = ((double)nchunk * (TH + 2) * pitch * p->rowb + (double)ni * bstage +
                         (double)TH * TW * npar * BN * 2) / 50.0;
    const double drain = ((nm * npar + 1) / 2) * (mask ? 50.0 : 30.0) * BN;
    const double cost = waves * (2000.0 + (occ > 1 ? std::max(drain + std::max(mma, copy), occ * std::max(mma, copy))
                                                    : drain + std::max(mma, copy)));
    if (cost >= best) return;
    best = cost;
    p->BN = BN;
    p->smem = smem;
    p->grid = dim3((unsigned)(B * tiles_x * tiles_y), (unsigned)(cout / BN));
    lbu::ConvTma& a = p->a;
    a.tiles_x = tiles_x;
    a.tiles_y = tiles_y;
    a.TH = TH;
    a.TW = TW;
    a.pitch = pitch;
    a.nm = nm;
    a.mstart = mstart;
    a.sbo = sbo;
    a.linear = linear ? 1 : 0;
    a.nchunk = nchunk;
    a.a_stride = a_stride;
    a.nstage = stages;
    a.cols = cols;
    a.tail = tail;
  };
  for (int BN = 128; BN >= 32; BN /= 2) {
    if (cout % BN) continue;
    for (int k = 1; k <= 8; k *= 2)
      if (8 * k < W + 8) consider(BN, 16, 8 * k, false);
    for (int TH = 1; TH <= 16 && TH <= H; ++TH) consider(BN, TH, std::min(W, 126), true);
  }
  return best < 1e30;
}

// Strips of conv3x3_rows_kernel over B images of H x W positions: wide images (at most a quarter
// of the 128-column strips' columns beyond the image, so W >= 96) whose weights for BN = 32 or 64
// output channels, with three input rows, fit in shared memory. More output channels are blocks of
// BN that each copy the input again. Every such layer takes the strips: this estimate and
// plan_tile's carry overheads fitted to their own kernel and are not comparable. Strips against
// tiles, us alone on the GPU, 32 images: 64 x 256, 32 -> 32 channels 20.9 / 29.3, 64 -> 32 29.2 /
// 60.6, 32 -> 64 37.2 / 59.2; 32 x 128, 128 -> 64 24.9 / 37.2; 32 x 96, 32 -> 32 10.9 / 16.7;
// 64 x 256 upsampled, 64 -> 32 28.4 / 41.5. One image: 64 x 256, 64 -> 32 8.7 / 10.5. Equal in
// several deep layers; slower where two blocks of 64 channels fill the chip: 32 x 128, 64 -> 128,
// 32 images 39.1 / 27.0 (8 images 12.8 / 13.0, one image 8.7 / 10.6). Two CTAs per multiprocessor where they fit, and the number
// of output rows per CTA with the smallest estimated time: waves of CTAs, each the longer of
// its MMAs (32 + N/4 cycles, N/2 above N = 128), its copies and its drain, and about 4,000
// cycles to start and end.
bool plan_rows(int B, int H, int W, int cin, int cout, int up, bool mask, ConvPlan* p) {
  const int tiles_x = (W + 127) / 128;
  if (4 * W < 3 * tiles_x * 128) return false;
  const int rowb = cin % 64 == 0 ? 128 : 64, nchunk = cin / (rowb / 2), npx = up ? 2 : 1, Ho = H << up;
  const int cstride = (130 * rowb + 1023) / 1024 * 1024;
  double best = 1e30;
  for (int BN = cout % 64 == 0 ? 64 : 32; BN >= 32; BN /= 2)
    for (int occ = 2; occ >= 1; --occ) {
      const int cols = 512 / occ;
      const int R = std::min(lbu::kRowsMaxSlot, cols / (npx * BN)) & ~1;
      if (R < 6) continue;  // three pairs: one drained, one completed, one begun
      const int weights = 9 * nchunk * BN * rowb, staging = 2 * 128 * BN * 2;
      const int room = kSmemSm / occ - 1024 - (int)sizeof(lbu::RowsTail) - 16 - weights - staging;
      int nrow = std::min(lbu::kRowsMaxStage, room / (nchunk * cstride));
      if (!up) nrow &= ~1;  // stages of two rows
      if (nrow < (up ? 3 : 4)) continue;
      const double n3 = 3 * BN, mma = 3.0 * nchunk * (rowb / 32) * npx * (n3 <= 128 ? 32 + n3 / 4 : n3 / 2);
      for (int TH = 2; TH <= Ho; TH += 2) {
        const int th = std::min(TH, Ho), tiles_h = (Ho + th - 1) / th;
        const double ctas = (double)B * tiles_x * tiles_h * (cout / BN);
        const double waves = std::ceil(ctas / (152.0 * occ));
        const double bytes = (double)(th / npx + 2) * nchunk * 130 * rowb + weights + (double)th * 128 * npx * BN * 2;
        const double drain = th / 2.0 * npx * BN * (mask ? 40.0 : 30.0);
        const double cost = waves * (4000.0 + weights / 50.0 + std::max(std::max(occ * (th + 2) * mma, occ * bytes / 50.0), drain));
        if (cost >= best) continue;
        best = cost;
        p->BN = BN;
        p->rowb = rowb;
        lbu::ConvRows& r = p->r;
        r.H = H;
        r.W = W;
        r.up = up;
        r.tiles_x = tiles_x;
        r.tiles_h = tiles_h;
        r.TH = th;
        r.nchunk = nchunk;
        r.cstride = cstride;
        r.nrow = nrow;
        r.R = R;
        r.cols = cols;
        r.w_off = nrow * nchunk * cstride;
        r.stg_off = r.w_off + weights;
        r.tail = r.stg_off + staging;
        // no more CTAs per SM than tensor memory serves
        p->smem = std::max(r.tail + (int)sizeof(lbu::RowsTail), kSmemSm / (occ + 1) - 1024 + 16);
        p->grid = dim3((unsigned)(B * tiles_x * tiles_h), (unsigned)(cout / BN));
      }
    }
  p->rows = best < 1e30;
  return p->rows;
}

ConvPlan conv_plan(const bf16* x, int xs, int B, int H, int W, int cin, int up, const bf16* w, const float* bias,
                   int relu, bf16* y, int ys, int cout, const bf16* mask, int ms) {
  ConvPlan p;
  if (cin % 32 || cout % 32 || xs % 8 || ys % 8 || ms % 8) return p;
  // whole 16-byte pieces are copied, loaded and stored
  if ((((uintptr_t)x | (uintptr_t)w | (uintptr_t)y | (uintptr_t)mask) & 15u) != 0) return p;
  const int Hi = H >> up, Wi = W >> up;
  if (plan_rows(B, Hi, Wi, cin, cout, up, mask != nullptr, &p)) {
    lbu::ConvRows& r = p.r;
    r.x = x;
    r.xs = xs;
    r.bias = bias;
    r.relu = relu;
    r.y = y;
    r.ys = ys;
    r.mask = mask;
    r.ms = ms;
    p.a.TW = 128;
    p.a.TH = -1;  // boxes of one row
  } else if (!plan_tile(B, Hi, Wi, cin, cout, up, mask != nullptr, &p)) {
    return p;
  }
  lbu::ConvTma& a = p.a;
  a.x = x;
  a.xs = xs;
  a.H = Hi;
  a.W = Wi;
  a.up = up;
  a.bias = bias;
  a.relu = relu;
  a.y = y;
  a.ys = ys;
  a.mask = mask;
  a.ms = ms;
  const cuuint32_t ch = (cuuint32_t)(p.rowb / 2);
  const cuuint64_t dx[4] = {(cuuint64_t)cin, (cuuint64_t)Wi, (cuuint64_t)Hi, (cuuint64_t)B};
  const cuuint64_t sx[3] = {(cuuint64_t)xs * 2, (cuuint64_t)Wi * xs * 2, (cuuint64_t)Hi * Wi * xs * 2};
  const cuuint32_t bx[4] = {ch, (cuuint32_t)a.TW + 2, (cuuint32_t)a.TH + 2, 1};
  const cuuint64_t dw[2] = {(cuuint64_t)9 * cin, (cuuint64_t)cout};
  const cuuint64_t sw[1] = {(cuuint64_t)9 * cin * 2};
  const cuuint32_t bw[2] = {ch, (cuuint32_t)p.BN};
  p.ok = encode_tiled(&p.mx, x, 4, dx, sx, bx, p.rowb) && encode_tiled(&p.mw, w, 2, dw, sw, bw, p.rowb);
  return p;
}

template <int BN, int ROWB>
cudaError_t launch_conv_tma(const ConvPlan& p, int* err, cudaStream_t s, bool chained) {
  static lbnci::SmemAllowance configured;
  cudaError_t e = lbnci::allow_smem(lbu::conv3x3_tma_kernel<BN, ROWB>, (size_t)p.smem, configured);
  if (e != cudaSuccess) return e;
  if (chained)
    return lbnci::launch_pdl(lbu::conv3x3_tma_kernel<BN, ROWB>, dim3(p.grid), dim3(lbu::kConvThreads), p.smem, s, p.mx,
                             p.mw, p.a, err);
  lbu::conv3x3_tma_kernel<BN, ROWB><<<p.grid, lbu::kConvThreads, p.smem, s>>>(p.mx, p.mw, p.a, err);
  return cudaGetLastError();
}
template <int BN, int ROWB>
cudaError_t launch_conv_rows(const ConvPlan& p, int* err, cudaStream_t s, bool chained) {
  static lbnci::SmemAllowance configured;
  cudaError_t e = lbnci::allow_smem(lbu::conv3x3_rows_kernel<BN, ROWB>, (size_t)p.smem, configured);
  if (e != cudaSuccess) return e;
  if (chained)
    return lbnci::launch_pdl(lbu::conv3x3_rows_kernel<BN, ROWB>, dim3(p.grid), dim3(lbu::kRowsThreads), p.smem, s, p.mx,
                             p.mw, p.r, err);
  lbu::conv3x3_rows_kernel<BN, ROWB><<<p.grid, lbu::kRowsThreads, p.smem, s>>>(p.mx, p.mw, p.r, err);
  return cudaGetLastError();
}
// chained: the launch follows a kernel of the network on its stream (whose wait the weights
// precede), so it may start while that one drains; a single convolution takes no part in it.
cudaError_t launch_conv_plan(const ConvPlan& p, int* err, cudaStream_t s, bool chained) {
  if (p.rows)
    return p.rowb == 128 ? (p.BN == 64 ? launch_conv_rows<64, 128>(p, err, s, chained) : launch_conv_rows<32, 128>(p, err, s, chained))
                         : (p.BN == 64 ? launch_conv_rows<64, 64>(p, err, s, chained) : launch_conv_rows<32, 64>(p, err, s, chained));
  if (p.rowb == 128)
    return p.BN == 128 ? launch_conv_tma<128, 128>(p, err, s, chained)
                       : (p.BN == 64 ? launch_conv_tma<64, 128>(p, err, s, chained) : launch_conv_tma<32, 128>(p, err, s, chained));
  return p.BN == 128 ? launch_conv_tma<128, 64>(p, err, s, chained)
                     : (p.BN == 64 ? launch_conv_tma<64, 64>(p, err, s, chained) : launch_conv_tma<32, 64>(p, err, s, chained));
}

// LBNCI_UNET_MMA=sync selects the mma.sync convolution and weight gradient for every layer. They
// stay for the layers whose input tile does not fit in shared memory (more than about 512
// channels) and for operands of single calls that are aligned to less than 16 bytes.
bool conv_on_mma_sync() {
  const char* e = std::getenv("LBNCI_UNET_MMA");
  return e && std::strcmp(e, "sync") == 0;
}

// Tensor maps of a weight gradient's operands: boxes of the tile and its ring (x) and of the
// tile (dy; when up, one map per parity of the output pixels).
bool wgrad_maps(lbu::WgradMaps* m, const WgradTmaPlan& p, const bf16* x, int xs, const bf16* dy, int dys, int B) {
  const lbu::WgradTma& a = p.a;
  const cuuint64_t W = (cuuint64_t)a.W, H = (cuuint64_t)a.H, b = (cuuint64_t)B;
  const cuuint64_t dx[4] = {(cuuint64_t)a.Cin, W, H, b};
  const cuuint64_t sx[3] = {(cuuint64_t)xs * 2, W * xs * 2, H * W * xs * 2};
  const cuuint32_t bx[4] = {(cuuint32_t)p.rowb / 2, (cuuint32_t)a.TW + 2, (cuuint32_t)a.TH + 2, 1};
  if (!encode_tiled(&m->x, x, 4, dx, sx, bx, p.rowb)) return false;
  const int f = a.up ? 2 : 1;
  const cuuint64_t dd[4] = {(cuuint64_t)a.Cout, W, H, b};
  const cuuint64_t sd[3] = {(cuuint64_t)f * dys * 2, (cuuint64_t)f * f * W * dys * 2, (cuuint64_t)f * f * H * W * dys * 2};
  const cuuint32_t bd[4] = {(cuuint32_t)p.BN, (cuuint32_t)a.TW, (cuuint32_t)a.TH, 1};
  for (int q = 0; q < 4; ++q) {
    const bf16* base = a.up ? dy + ((size_t)(q >> 1) * f * W + (q & 1)) * dys : dy;
    if (!encode_tiled(&m->dy[q], base, 4, dd, sd, bd, p.BN * 2)) return false;
  }
  return true;
}

template <int BN, int ROWB>
cudaError_t launch_wgrad_tma(const WgradTmaPlan& p, const lbu::WgradMaps& maps, int* err, cudaStream_t s) {
  static lbnci::SmemAllowance configured;
  cudaError_t e = lbnci::allow_smem(lbu::conv3x3_wgrad_tma_kernel<BN, ROWB>, (size_t)p.smem, configured);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)p.a.nsplit, (unsigned)(p.a.Cin / (ROWB / 2)), (unsigned)(p.a.Cout / BN));
  lbnci::launch_pdl(lbu::conv3x3_wgrad_tma_kernel<BN, ROWB>, grid, dim3(lbu::kConvThreads), p.smem, s, maps, p.a, err);
  return cudaGetLastError();
}

// The error word of a launch: the network's, or that of the single calls.
cudaError_t error_word(lbu_net* n, int** err) {
  if (n) {
    *err = n->tc_err;
    return cudaSuccess;
  }
  g_single_used = true;
  return cudaGetSymbolAddress((void**)err, g_tc_err);
}

// Test of the reporting (never set in use): LBNCI_UNET_FAIL_TEST=1 sets the error word behind
// every tensor-core launch, as a kernel whose wait ran out would.
cudaError_t fail_test(int* err, cudaStream_t s) {
  const char* e = std::getenv("LBNCI_UNET_FAIL_TEST");
  return e && std::atoi(e) == 1 ? cudaMemsetAsync(err, 1, sizeof(int), s) : cudaSuccess;
}

// Synchronises the network's stream, reports and clears an expired wait of its kernels, and
// returns the loss. An expired wait of a single call is reported too, after the results.
lb_status finish(lbu_net* n, float* loss) {
  Report r;
  cudaError_t e = cudaMemcpyAsync(&r, n->loss, sizeof(r), cudaMemcpyDeviceToHost, n->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
  if (e != cudaSuccess) return cuda_fail(n, e, "result read");
  if (r.err) {
    e = cudaMemsetAsync(n->tc_err, 0, 2 * sizeof(int), n->stream);
    if (e != cudaSuccess) return cuda_fail(n, e, "error word reset");
    n->t -= r.skipped;
    return fail(n, LB_ECUDA, "a tensor-core convolution's mbarrier wait expired (no output written; " +
                                 std::to_string(r.skipped) + " parameter updates left out since)");
  }
  if (loss) *loss = (float)r.loss;
  if (!g_single_used) return LB_OK;
  int v = 0;
  e = cudaMemcpyFromSymbol(&v, g_tc_err, sizeof(int));
  if (e != cudaSuccess) return cuda_fail(n, e, "error word read");
  if (v) {
    const int zero = 0;
    cudaMemcpyToSymbol(g_tc_err, &zero, sizeof(int));
    return fail(n, LB_ECUDA, "an earlier single convolution's (lbu_conv3x3, lbu_conv3x3_wgrad) mbarrier wait expired, "
                             "it wrote no output; this call's results are complete");
  }
  return LB_OK;
}

// one 3x3 convolution launch (forward or data gradient); site: the network's cache slot
lb_status conv(lbu_net* n, int site, const bf16* x, int xs, int B, int H, int W, int cin, int up, const bf16* w,
               const float* bias, int relu, bf16* y, int ys, int cout, const bf16* mask, int ms,
               cudaStream_t s) {
  if (!conv_on_mma_sync()) {
    ConvCache once;
    ConvCache& c = n ? n->conv_cache[site] : once;
    if (c.B != B) {
      c.p = conv_plan(x, xs, B, H, W, cin, up, w, bias, relu, y, ys, cout, mask, ms);
      c.B = B;
    }
    if (c.p.ok) {
      int* err = nullptr;
      cudaError_t e = error_word(n, &err);
      if (e == cudaSuccess) e = launch_conv_plan(c.p, err, s, n != nullptr);
      if (e == cudaSuccess) e = fail_test(err, s);
      if (n) ++n->launches;
      return e == cudaSuccess ? LB_OK : cuda_fail(n, e, "conv3x3 (tensor memory) launch");
    }
  }
  lbu::ConvFwd a{x, xs, B, H, W, cin, up, w, bias, relu, y, ys, cout, mask, ms};
  const int M = B * H * W;
  dim3 grid((M + lbu::kConvBM - 1) / lbu::kConvBM, 1);
  if (cout % 64 == 0) {
    grid.y = cout / 64;
    lbu::conv3x3_kernel<64><<<grid, 128, 0, s>>>(a);
  } else {
    grid.y = cout / 32;
    lbu::conv3x3_kernel<32><<<grid, 128, 0, s>>>(a);
  }
  if (n) ++n->launches;
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LB_OK : cuda_fail(n, e, "conv3x3 launch");
}

lb_status wgrad(lbu_net* n, int site, const bf16* x, int xs, int up, const bf16* dy, int dys, int B, int H, int W, int cin,
                int cout, float* work, size_t work_bytes, cudaStream_t s, float* dw_master, float* db_master,
                int cin_true) {
  // 16-byte pieces of x and dy are copied, and the reduction loads the partial sums in work as such
  if (!conv_on_mma_sync() && xs % 8 == 0 && dys % 8 == 0 &&
      (((uintptr_t)x | (uintptr_t)dy | (uintptr_t)work) & 15u) == 0) {
    WgradCache once;
    WgradCache& c = n ? n->wgrad_cache[site] : once;
    if (c.B != B) {
      c.p = wgrad_tma_plan(B, H >> up, W >> up, cin, cout, up);
      c.p.ok = c.p.ok && wgrad_maps(&c.maps, c.p, x, xs, dy, dys, B);
      c.B = B;
    }
    WgradTmaPlan& p = c.p;
    const lbu::WgradMaps& maps = c.maps;
    if (p.ok && wgrad_tma_bytes(p) <= work_bytes) {
      p.a.x = x;
      p.a.xs = xs;
      p.a.part = work;
      float* bp = work + (size_t)p.a.nsplit * cout * (up ? 16 : 9) * cin;
      p.a.bpart = db_master ? bp : nullptr;
      int* err = nullptr;
      cudaError_t e = error_word(n, &err);
      if (e == cudaSuccess)
        e = p.rowb == 128 ? (p.BN == 64 ? launch_wgrad_tma<64, 128>(p, maps, err, s)
                                        : launch_wgrad_tma<32, 128>(p, maps, err, s))
                          : (p.BN == 64 ? launch_wgrad_tma<64, 64>(p, maps, err, s)
                                        : launch_wgrad_tma<32, 64>(p, maps, err, s));
      if (e == cudaSuccess) e = fail_test(err, s);
      if (e != cudaSuccess) return cuda_fail(n, e, "wgrad (tensor memory) launch");
      const int n4 = cout * 9 * cin / 4;
      int S = 1;  // threads to each group of four values: about four blocks per multiprocessor
      while (S < 32 && 2 * S <= p.a.nsplit && (long long)n4 * S < 152LL * 4 * 256) S *= 2;
      const int wblocks = (n4 + 256 / S - 1) / (256 / S), bblocks = db_master ? (cout + 31) / 32 : 0;
      lbnci::launch_pdl(lbu::wgrad_reduce_tma_kernel, dim3(wblocks + bblocks), dim3(256), 0, s, work, bp, p.a.nsplit,
                        cout, cin, cin_true, up, S, wblocks, dw_master, db_master);
      if (n) n->launches += 2;
      e = cudaGetLastError();
      return e == cudaSuccess ? LB_OK : cuda_fail(n, e, "wgrad reduction launch");
    }
  }
  const WgradPlan p = wgrad_plan(B * H * W, cin, cout);
  if (wgrad_bytes(p, cin, cout) > work_bytes) return fail(n, LB_EINVAL, "wgrad scratch too small");
  float* part = work;
  float* bpart = work + (size_t)p.nsplit * cout * 9 * cin;
  lbu::ConvWgrad a{x, xs, up, dy, dys, B, H, W, cin, cout, part, db_master ? bpart : nullptr, p.pps};
  dim3 grid(cout / p.BM, 9 * (cin / p.BN), p.nsplit);
  if (p.BM == 64 && p.BN == 64) lbu::conv3x3_wgrad_kernel<64, 64><<<grid, 128, 0, s>>>(a);
  else if (p.BM == 64) lbu::conv3x3_wgrad_kernel<64, 32><<<grid, 128, 0, s>>>(a);
  else if (p.BN == 64) lbu::conv3x3_wgrad_kernel<32, 64><<<grid, 128, 0, s>>>(a);
  else lbu::conv3x3_wgrad_kernel<32, 32><<<grid, 128, 0, s>>>(a);
  const long long nout = (long long)cout * 9 * cin_true + cout;
  lbu::wgrad_reduce_kernel<<<grid_for(nout, 256), 256, 0, s>>>(part, bpart, p.nsplit, cout, cin, cin_true,
                                                                dw_master, db_master);
  if (n) n->launches += 2;
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LB_OK : cuda_fail(n, e, "wgrad launch");
}

#define LBU_TRY(expr)                  \
  do {                                 \
    lb_status st_ = (expr);            \
    if (st_ != LB_OK) return st_;      \
  } while (0)

const bf16* WB(const lbu_net* n, int i) { return n->wb + n->L[i].wb_off; }
const bf16* WT(const lbu_net* n, int i) { return n->wt + n->L[i].wt_off; }
const float* BIAS(const lbu_net* n, int i) { return n->params + n->L[i].b_off; }

// index helpers into the layer table
int enc_a(int l) { return 2 * l; }
int enc_b(int l) { return 2 * l + 1; }
int up_i(const lbu_net* n, int l) { return 2 * n->cfg.levels + 3 * (n->cfg.levels - 2 - l); }
int head_i(const lbu_net* n) { return (int)n->L.size() - 1; }

// The head's kernels are built for each number of outputs.
template <typename F>
void for_outputs(int nout, F&& f) {
  static_assert(lbu::kMaxOut == 8, "one build per number of outputs");
  switch (nout) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    case 5: return f(std::integral_constant<int, 5>{});
    case 6: return f(std::integral_constant<int, 6>{});
    case 7: return f(std::integral_constant<int, 7>{});
    default: return f(std::integral_constant<int, 8>{});
  }
}

lb_status forward_impl(lbu_net* n, int B) {
  const int Lv = n->cfg.levels;
  cudaStream_t s = n->stream;
  const bf16* h = n->x0;
  int hs = kInPad;
  for (int l = 0; l < Lv; ++l) {
    const int C = width(n, l), H = Hl(n, l), W = Wl(n, l);
    LBU_TRY(conv(n, enc_a(l), h, hs, B, H, W, n->L[enc_a(l)].cin_pad, 0, WB(n, enc_a(l)), BIAS(n, enc_a(l)), 1, n->ea[l], C,
                 C, nullptr, 0, s));
    if (l < Lv - 1) {
      LBU_TRY(conv(n, enc_b(l), n->ea[l], C, B, H, W, C, 0, WB(n, enc_b(l)), BIAS(n, enc_b(l)), 1, n->cat[l] + C, 2 * C, C,
                   nullptr, 0, s));
      const long long work = (long long)B * (H / 2) * (W / 2) * (C / 8);
      lbnci::launch_pdl(lbu::maxpool_kernel, dim3(grid_for(work, 256)), dim3(256), 0, s,
                        n->cat[l] + C, 2 * C, B, H, W, C, n->pool[l]);
      ++n->launches;
      h = n->pool[l];
      hs = C;
    } else {
      LBU_TRY(conv(n, enc_b(l), n->ea[l], C, B, H, W, C, 0, WB(n, enc_b(l)), BIAS(n, enc_b(l)), 1, n->db[l], C, C, nullptr,
                   0, s));
      h = n->db[l];
      hs = C;
    }
  }
  for (int l = Lv - 2; l >= 0; --l) {
    const int C = width(n, l), H = Hl(n, l), W = Wl(n, l), k = up_i(n, l);
    LBU_TRY(conv(n, k, h, hs, B, H, W, 2 * C, 1, WB(n, k), BIAS(n, k), 1, n->cat[l], 2 * C, C, nullptr, 0, s));
    LBU_TRY(conv(n, k + 1, n->cat[l], 2 * C, B, H, W, 2 * C, 0, WB(n, k + 1), BIAS(n, k + 1), 1, n->da[l], C, C, nullptr,
                 0, s));
    LBU_TRY(conv(n, k + 2, n->da[l], C, B, H, W, C, 0, WB(n, k + 2), BIAS(n, k + 2), 1, n->db[l], C, C, nullptr, 0, s));
    h = n->db[l];
    hs = C;
  }
  const int hi = head_i(n);
  const int P = B * n->cfg.H * n->cfg.W;
  for_outputs(n->cfg.out_ch, [&](auto NOUT) {
    lbnci::launch_pdl(lbu::head_fwd_kernel<decltype(NOUT)::value>, dim3(grid_for(P, 256)), dim3(256), 0, s, n->db[0],
                      n->cfg.base, WB(n, hi), BIAS(n, hi), P, n->y);
  });
  ++n->launches;
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LB_OK : cuda_fail(n, e, "forward launch");
}

lb_status backward_impl(lbu_net* n, int B) {
  const int Lv = n->cfg.levels;
  cudaStream_t s = n->stream;
  const int P = B * n->cfg.H * n->cfg.W;
  const int nl = (int)n->L.size();
  float* G = n->grads;
  auto GW = [&](int i) { return G + n->L[i].w_off; };
  auto GB = [&](int i) { return G + n->L[i].b_off; };
  // head
  {
    const int hi = head_i(n), C0 = n->cfg.base;
    const int nblk = (P + lbu::kHeadPix - 1) / lbu::kHeadPix;
    for_outputs(n->cfg.out_ch, [&](auto NOUT) {
      lbnci::launch_pdl(lbu::head_bwd_kernel<decltype(NOUT)::value>, dim3(nblk), dim3(256), 0, s, n->db[0], C0,
                        WB(n, hi), P, n->dy, n->gB[0], n->work);
    });
    lbnci::launch_pdl(lbu::head_reduce_kernel,
                      dim3(n->cfg.out_ch * (C0 + 1)), dim3(128), 0, s, n->work, nblk, n->cfg.out_ch, C0, GW(hi), GB(hi));
    n->launches += 2;
  }
  // decoder, finest level first
  for (int l = 0; l <= Lv - 2; ++l) {
    const int C = width(n, l), H = Hl(n, l), W = Wl(n, l), k = up_i(n, l);
    const int C1 = width(n, l + 1);
    // dec_lb: input da[l], output gradient gB[l]
    LBU_TRY(wgrad(n, k + 2, n->da[l], C, 0, n->gB[l], C, B, H, W, C, C, n->work, n->work_bytes, s, GW(k + 2), GB(k + 2), C));
    LBU_TRY(conv(n, nl + k + 2, n->gB[l], C, B, H, W, C, 0, WT(n, k + 2), nullptr, 0, n->gA[l], C, C, n->da[l], C, s));
    // dec_la: input cat[l]
    LBU_TRY(wgrad(n, k + 1, n->cat[l], 2 * C, 0, n->gA[l], C, B, H, W, 2 * C, C, n->work, n->work_bytes, s, GW(k + 1),
                  GB(k + 1), 2 * C));
    LBU_TRY(conv(n, nl + k + 1, n->gA[l], C, B, H, W, C, 0, WT(n, k + 1), nullptr, 0, n->gCat[l], 2 * C, 2 * C, n->cat[l],
                 2 * C, s));
    // up_l: input = nearest upsampling of the level-(l+1) output
    const bf16* hin = n->db[l + 1];
    LBU_TRY(wgrad(n, k, hin, C1, 1, n->gCat[l], 2 * C, B, H, W, C1, C, n->work, n->work_bytes, s, GW(k), GB(k), C1));
    LBU_TRY(conv(n, nl + k, n->gCat[l], 2 * C, B, H, W, C, 0, WT(n, k), nullptr, 0, n->gU[l], C1, C1, nullptr, 0, s));
    const long long work = (long long)B * Hl(n, l + 1) * Wl(n, l + 1) * (C1 / 8);
    lbnci::launch_pdl(lbu::upsample_bwd_kernel, dim3(grid_for(work, 256)), dim3(256), 0, s,
                      n->gU[l], hin, n->gB[l + 1], B, Hl(n, l + 1), Wl(n, l + 1), C1);
    ++n->launches;
  }
  // encoder, coarsest level first; gB[Lv-1] holds the bottom output's gradient
  for (int l = Lv - 1; l >= 0; --l) {
    const int C = width(n, l), H = Hl(n, l), W = Wl(n, l);
    const bf16* g;
    int gs;
    if (l == Lv - 1) {
      g = n->gB[l];
      gs = C;
    } else {
      const long long work = (long long)B * (H / 2) * (W / 2) * (C / 8);
      lbnci::launch_pdl(lbu::maxpool_bwd_kernel, dim3(grid_for(work, 256)), dim3(256), 0, s,
                        n->cat[l] + C, 2 * C, n->gPool[l], n->gCat[l] + C, 2 * C, B, H, W, C);
      ++n->launches;
      g = n->gCat[l] + C;
      gs = 2 * C;
    }
    LBU_TRY(wgrad(n, enc_b(l), n->ea[l], C, 0, g, gs, B, H, W, C, C, n->work, n->work_bytes, s, GW(enc_b(l)), GB(enc_b(l)), C));
    LBU_TRY(conv(n, nl + enc_b(l), g, gs, B, H, W, C, 0, WT(n, enc_b(l)), nullptr, 0, n->gA[l], C, C, n->ea[l], C, s));
    const bf16* xin = l == 0 ? n->x0 : n->pool[l - 1];
    const int cin = n->L[enc_a(l)].cin_pad;
    LBU_TRY(wgrad(n, enc_a(l), xin, cin, 0, n->gA[l], C, B, H, W, cin, C, n->work, n->work_bytes, s, GW(enc_a(l)),
                  GB(enc_a(l)), n->L[enc_a(l)].cin));
    if (l > 0)
      LBU_TRY(conv(n, nl + enc_a(l), n->gA[l], C, B, H, W, C, 0, WT(n, enc_a(l)), nullptr, 0, n->gPool[l - 1], cin, cin, nullptr,
                   0, s));
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LB_OK : cuda_fail(n, e, "backward launch");
}

lb_status refresh(lbu_net* n) {
  size_t maxn = 0;
  for (auto& l : n->L) maxn = std::max(maxn, (size_t)l.cout * l.taps * l.cin_pad);
  dim3 grid((unsigned)std::min<size_t>((maxn + 255) / 256, 1024), (unsigned)n->L.size());
  lbnci::launch_pdl(lbu::refresh_weights_kernel, grid, dim3(256), 0, n->stream, n->Ldev, n->params, n->wb, n->wt);
  ++n->launches;
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LB_OK : cuda_fail(n, e, "refresh launch");
}

lb_status loss_impl(lbu_net* n, const float* T, const int* idx, int B, const float* lam) {
  const int HW = n->cfg.H * n->cfg.W, P = B * HW;
  float lm[8];
  for (int j = 0; j < 8; ++j) lm[j] = (lam && j < n->cfg.out_ch) ? lam[j] : 1.f;
  const int blocks = std::min(n->npartial, grid_for(P, 256));
  lbnci::launch_pdl(lbu::mse_kernel, dim3(blocks), dim3(256), 0, n->stream, n->y, T, idx, HW, n->cfg.out_ch, P, lm[0],
                    lm[1], lm[2], lm[3], lm[4], lm[5], lm[6], lm[7], n->dy, n->partial);
  lbnci::launch_pdl(lbu::sum_partials_kernel, dim3(1), dim3(256), 0, n->stream, n->partial, blocks, 1.0 / P, n->loss);
  n->launches += 2;
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LB_OK : cuda_fail(n, e, "loss launch");
}

lb_status pack(lbu_net* n, const float* X, const int* idx, int B) {
  const long long work = (long long)B * n->cfg.H * n->cfg.W * (kInPad / 8);
  lbnci::launch_pdl(lbu::pack_input_kernel, dim3(grid_for(work, 256)), dim3(256), 0,
                    n->stream, X, idx, B, n->cfg.H * n->cfg.W, n->cfg.in_ch, kInPad, n->x0);
  ++n->launches;
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LB_OK : cuda_fail(n, e, "pack launch");
}

// Whether p is a multiple of n bytes. Both convolution kernels copy x, the weights and dy in
// 16-byte pieces (mma.sync by cp.async), mma.sync stores pairs of channels and pairs of partial
// sums: a pointer below that alignment is refused, no kernel could take it.
bool aligned(const void* p, unsigned n) { return ((uintptr_t)p & (n - 1u)) == 0; }

lb_status check_batch(lbu_net* n, int B) {
  if (B <= 0 || B > n->cfg.max_batch) return fail(n, LB_EINVAL, "batch must be 1..max_batch");
  return LB_OK;
}

}  // namespace

extern "C" {

int lbu_layer_count(const lbu_config* cfg) {
  std::string why;
  if (!valid_config(cfg, &why)) return -1;
  return (int)layer_table(cfg).size();
}

lb_status lbu_layer_shape(const lbu_config* cfg, int layer, int shape[4]) {
  std::string why;
  if (!valid_config(cfg, &why)) return fail(nullptr, LB_EINVAL, why);
  auto L = layer_table(cfg);
  if (layer < 0 || layer >= (int)L.size() || !shape) return fail(nullptr, LB_EINVAL, "bad layer index");
  const int k = L[layer].taps == 9 ? 3 : 1;
  shape[0] = L[layer].cout;
  shape[1] = k;
  shape[2] = k;
  shape[3] = L[layer].cin;
  return LB_OK;
}

lb_status lbu_param_count(const lbu_config* cfg, long long* count) {
  std::string why;
  if (!valid_config(cfg, &why)) return fail(nullptr, LB_EINVAL, why);
  if (!count) return fail(nullptr, LB_EINVAL, "null count");
  *count = total_params(layer_table(cfg));
  return LB_OK;
}

lb_status lbu_create(const lbu_config* cfg, lbu_net** out) {
  std::string why;
  if (!out) return fail(nullptr, LB_EINVAL, "null output handle");
  *out = nullptr;
  if (!valid_config(cfg, &why)) return fail(nullptr, LB_EINVAL, why);
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
    (void)cudaGetLastError();
    return fail(nullptr, LB_ECUDA, "no CUDA device");
  }
  lbu_net* n = new (std::nothrow) lbu_net();
  if (!n) return fail(nullptr, LB_ENOMEM, "host allocation failed");
  n->cfg = *cfg;
  n->stream = (cudaStream_t)cfg->stream;
  cudaGetDevice(&n->device);
  n->L = layer_table(cfg);
  n->nparams = total_params(n->L);
  n->conv_cache.resize(2 * n->L.size());
  n->wgrad_cache.resize(n->L.size());
  const int Lv = cfg->levels, B = cfg->max_batch;
  auto bail = [&](lb_status st) {
    g_err = n->err;
    lbu_destroy(n);
    return st;
  };
#define LBU_ALLOC(p, cnt)                          \
  do {                                             \
    lb_status st_ = dalloc(n, &(p), (cnt));        \
    if (st_ != LB_OK) return bail(st_);            \
  } while (0)
  LBU_ALLOC(n->params, n->nparams);
  LBU_ALLOC(n->grads, n->nparams);
  LBU_ALLOC(n->m, n->nparams);
  LBU_ALLOC(n->v, n->nparams);
  long long nwb = 0, nwt = 0;
  for (auto& l : n->L) {
    nwb = std::max(nwb, l.wb_off + (long long)l.cout * l.taps * l.cin_pad);
    if (l.wt_off >= 0) nwt = std::max(nwt, l.wt_off + (long long)l.cout * 9 * l.cin_pad);
  }
  LBU_ALLOC(n->wb, nwb);
  LBU_ALLOC(n->wt, nwt);
  LBU_ALLOC(n->Ldev, n->L.size());
  {
    std::vector<lbu::LayerDev> h(n->L.size());
    for (size_t i = 0; i < n->L.size(); ++i) {
      const LayerHost& l = n->L[i];
      h[i] = lbu::LayerDev{l.w_off, l.b_off, l.wb_off, l.wt_off, l.cout, l.cin, l.cin_pad, l.taps};
    }
    if (cudaMemcpy(n->Ldev, h.data(), h.size() * sizeof(h[0]), cudaMemcpyHostToDevice) != cudaSuccess)
      return bail(cuda_fail(n, cudaGetLastError(), "layer table copy"));
  }
  const size_t HW = (size_t)cfg->H * cfg->W;
  n->ea.assign(Lv, nullptr);
  n->cat.assign(Lv, nullptr);
  n->pool.assign(Lv, nullptr);
  n->da.assign(Lv, nullptr);
  n->db.assign(Lv, nullptr);
  n->gA.assign(Lv, nullptr);
  n->gB.assign(Lv, nullptr);
  n->gCat.assign(Lv, nullptr);
  n->gU.assign(Lv, nullptr);
  n->gPool.assign(Lv, nullptr);
  for (int l = 0; l < Lv; ++l) {
    const size_t pix = (size_t)B * (HW >> (2 * l));
    const int C = width(n, l);
    LBU_ALLOC(n->ea[l], pix * C);
    LBU_ALLOC(n->db[l], pix * C);
    LBU_ALLOC(n->gA[l], pix * C);
    LBU_ALLOC(n->gB[l], pix * C);
    if (l < Lv - 1) {
      LBU_ALLOC(n->cat[l], pix * 2 * C);
      LBU_ALLOC(n->gCat[l], pix * 2 * C);
      LBU_ALLOC(n->da[l], pix * C);
      LBU_ALLOC(n->pool[l], (pix / 4) * C);
      LBU_ALLOC(n->gPool[l], (pix / 4) * C);
      LBU_ALLOC(n->gU[l], pix * width(n, l + 1));
    }
  }
  LBU_ALLOC(n->x0, (size_t)B * HW * kInPad);
  LBU_ALLOC(n->y, (size_t)B * HW * cfg->out_ch);
  LBU_ALLOC(n->dy, (size_t)B * HW * cfg->out_ch);
  LBU_ALLOC(n->xstage, (size_t)B * HW * cfg->in_ch);
  LBU_ALLOC(n->ystage, (size_t)B * HW * cfg->out_ch);
  // scratch: the largest wgrad partial set and the head partials
  size_t wb = 0;
  for (int l = 0; l < Lv; ++l) {
    const int C = width(n, l);
    const int cins[4] = {l == 0 ? kInPad : width(n, l - 1), C, 2 * C, l < Lv - 1 ? width(n, l + 1) : C};
    for (int ci : cins) wb = std::max(wb, wgrad_work(B, Hl(n, l), Wl(n, l), ci, C));
  }
  const size_t nblk = ((size_t)B * HW + lbu::kHeadPix - 1) / lbu::kHeadPix;
  wb = std::max(wb, nblk * cfg->out_ch * (cfg->base + 1) * sizeof(float));
  n->work_bytes = wb;
  LBU_ALLOC(n->work, wb / sizeof(float) + 1);
  n->npartial = 152 * 16;
  LBU_ALLOC(n->partial, n->npartial);
  LBU_ALLOC(n->loss, sizeof(Report) / sizeof(double));
  n->tc_err = &reinterpret_cast<Report*>(n->loss)->err;
#undef LBU_ALLOC
  if (cudaMemset(n->params, 0, n->nparams * sizeof(float)) != cudaSuccess ||
      cudaMemset(n->m, 0, n->nparams * sizeof(float)) != cudaSuccess ||
      cudaMemset(n->v, 0, n->nparams * sizeof(float)) != cudaSuccess ||
      cudaMemset(n->grads, 0, n->nparams * sizeof(float)) != cudaSuccess ||
      cudaMemset(n->loss, 0, sizeof(Report)) != cudaSuccess)
    return bail(cuda_fail(n, cudaGetLastError(), "cudaMemset"));
  if (refresh(n) != LB_OK || cudaStreamSynchronize(n->stream) != cudaSuccess)
    return bail(cuda_fail(n, cudaGetLastError(), "initial weight refresh"));
  *out = n;
  return LB_OK;
}

void lbu_destroy(lbu_net* n) {
  if (!n) return;
  if (n->stream) cudaStreamSynchronize(n->stream);
  else cudaDeviceSynchronize();
  for (void* p : n->allocs) cudaFree(p);
  (void)cudaGetLastError();
  delete n;
}

const char* lbu_last_error(const lbu_net* n) { return n ? n->err.c_str() : g_err.c_str(); }

long long lbu_kernel_launches(const lbu_net* n) { return n ? n->launches : 0; }

lb_status lbu_set_params(lbu_net* n, const float* p, int on_device) {
  if (!n || !p) return fail(n, LB_EINVAL, "null argument");
  LBU_CUDA(n, cudaMemcpyAsync(n->params, p, n->nparams * sizeof(float),
                              on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, n->stream));
  LBU_CUDA(n, cudaMemsetAsync(n->m, 0, n->nparams * sizeof(float), n->stream));
  LBU_CUDA(n, cudaMemsetAsync(n->v, 0, n->nparams * sizeof(float), n->stream));
  LBU_CUDA(n, cudaMemsetAsync(n->tc_err + 1, 0, sizeof(int), n->stream));  // Report::skipped
  n->t = 0;
  LBU_TRY(refresh(n));
  LBU_CUDA(n, cudaStreamSynchronize(n->stream));
  return LB_OK;
}

lb_status lbu_get_params(lbu_net* n, float* p, int on_device) {
  if (!n || !p) return fail(n, LB_EINVAL, "null argument");
  LBU_CUDA(n, cudaMemcpyAsync(p, n->params, n->nparams * sizeof(float),
                              on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, n->stream));
  LBU_CUDA(n, cudaStreamSynchronize(n->stream));
  return LB_OK;
}

lb_status lbu_set_adam(lbu_net* n, float b1, float b2, float eps) {
  if (!n) return fail(n, LB_EINVAL, "null handle");
  if (!(b1 >= 0.f && b1 < 1.f && b2 >= 0.f && b2 < 1.f && eps > 0.f)) return fail(n, LB_EINVAL, "bad Adam parameters");
  n->b1 = b1;
  n->b2 = b2;
  n->eps = eps;
  return LB_OK;
}

lb_status lbu_forward(lbu_net* n, const float* x, int batch, float* y, int on_device) {
  if (!n || !x || !y) return fail(n, LB_EINVAL, "null argument");
  LBU_TRY(check_batch(n, batch));
  const size_t HW = (size_t)n->cfg.H * n->cfg.W;
  const float* xd = x;
  if (!on_device) {
    LBU_CUDA(n, cudaMemcpyAsync(n->xstage, x, batch * HW * n->cfg.in_ch * sizeof(float), cudaMemcpyHostToDevice,
                                n->stream));
    xd = n->xstage;
  }
  LBU_TRY(pack(n, xd, nullptr, batch));
  LBU_TRY(forward_impl(n, batch));
  LBU_CUDA(n, cudaMemcpyAsync(y, n->y, batch * HW * n->cfg.out_ch * sizeof(float),
                              on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, n->stream));
  return on_device ? LB_OK : finish(n, nullptr);
}

lb_status lbu_loss_grad(lbu_net* n, const float* X, const float* T, const int* idx, int batch, const float* lam,
                        float* loss, float* grads) {
  if (!n || !X || !T) return fail(n, LB_EINVAL, "null argument");
  LBU_TRY(check_batch(n, batch));
  LBU_TRY(pack(n, X, idx, batch));
  LBU_TRY(forward_impl(n, batch));
  LBU_TRY(loss_impl(n, T, idx, batch, lam));
  LBU_TRY(backward_impl(n, batch));
  if (grads)
    LBU_CUDA(n, cudaMemcpyAsync(grads, n->grads, n->nparams * sizeof(float), cudaMemcpyDeviceToDevice, n->stream));
  return loss ? finish(n, loss) : LB_OK;
}

lb_status lbu_train_step(lbu_net* n, const float* X, const float* T, const int* idx, int batch, const float* lam,
                         float lr, float* loss) {
  if (!n) return fail(n, LB_EINVAL, "null handle");
  if (!(lr > 0.f)) return fail(n, LB_EINVAL, "learning rate must be positive");
  LBU_TRY(lbu_loss_grad(n, X, T, idx, batch, lam, nullptr, nullptr));
  ++n->t;
  const float c1 = (float)(1.0 / (1.0 - std::pow((double)n->b1, (double)n->t)));
  const float c2 = (float)(1.0 / (1.0 - std::pow((double)n->b2, (double)n->t)));
  lbnci::launch_pdl(lbu::adam_kernel, dim3(grid_for(n->nparams, 256)), dim3(256), 0, n->stream, n->params, n->grads,
                    n->m, n->v, n->nparams, lr, n->b1, n->b2, n->eps, c1, c2, n->tc_err);
  ++n->launches;
  LBU_CUDA(n, cudaGetLastError());
  LBU_TRY(refresh(n));
  return loss ? finish(n, loss) : LB_OK;
}

lb_status lbu_conv3x3(const unsigned short* x, int x_stride, int batch, int h, int w, int c_in, int upsample,
                      const unsigned short* wgt, const float* bias, int relu, unsigned short* y, int y_stride,
                      int c_out, void* stream) {
  if (!x || !wgt || !y) return fail(nullptr, LB_EINVAL, "null argument");
  if (batch <= 0 || h <= 0 || w <= 0 || c_in <= 0 || c_out <= 0 || c_in % 32 || c_out % 32)
    return fail(nullptr, LB_EINVAL, "sizes: positive, channels multiples of 32");
  if (x_stride < c_in || y_stride < c_out || x_stride % 8 || y_stride % 8)
    return fail(nullptr, LB_EINVAL, "strides: at least the channel count, multiples of 8");
  if (!aligned(x, 16) || !aligned(wgt, 16) || !aligned(y, 4))
    return fail(nullptr, LB_EINVAL, "alignment: x and weights 16 bytes, y 4 bytes");
  if (upsample && (h % 2 || w % 2)) return fail(nullptr, LB_EINVAL, "upsampled output must have even size");
  return conv(nullptr, 0, (const bf16*)x, x_stride, batch, h, w, c_in, upsample ? 1 : 0, (const bf16*)wgt, bias, relu,
              (bf16*)y, y_stride, c_out, nullptr, 0, (cudaStream_t)stream);
}

size_t lbu_conv3x3_wgrad_work(int batch, int h, int w, int c_in, int c_out) {
  if (batch <= 0 || h <= 0 || w <= 0 || c_in <= 0 || c_out <= 0) return 0;
  return wgrad_work(batch, h, w, c_in, c_out);
}

lb_status lbu_conv3x3_wgrad(const unsigned short* x, int x_stride, int batch, int h, int w, int c_in, int upsample,
                            const unsigned short* dy, int dy_stride, int c_out, float* dw, float* db, void* work,
                            size_t work_bytes, void* stream) {
  if (!x || !dy || !dw || !work) return fail(nullptr, LB_EINVAL, "null argument");
  if (batch <= 0 || h <= 0 || w <= 0 || c_in % 32 || c_out % 32 || c_in <= 0 || c_out <= 0)
    return fail(nullptr, LB_EINVAL, "sizes: positive, channels multiples of 32");
  if (x_stride < c_in || dy_stride < c_out || x_stride % 8 || dy_stride % 8)
    return fail(nullptr, LB_EINVAL, "strides: at least the channel count, multiples of 8");
  if (!aligned(x, 16) || !aligned(dy, 16) || !aligned(work, 8))
    return fail(nullptr, LB_EINVAL, "alignment: x and dy 16 bytes, work 8 bytes");
  if (upsample && (h % 2 || w % 2)) return fail(nullptr, LB_EINVAL, "upsampled output must have even size");
  return wgrad(nullptr, 0, (const bf16*)x, x_stride, upsample ? 1 : 0, (const bf16*)dy, dy_stride, batch, h, w, c_in,
               c_out, (float*)work, work_bytes, (cudaStream_t)stream, dw, db, c_in);
}

}  // extern "C"
