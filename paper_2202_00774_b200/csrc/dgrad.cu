// Host side of the data-gradient contraction: tensor maps, tile shapes, the choice of kernel (see dgrad_general.cu and
// dgrad_halo.cuh for the kernels).
#include <string.h>

#include <algorithm>
#include <iterator>

#include "dgrad_general.cuh"
#include "dgrad_halo_params.cuh"
#include "dgrad_rows.cuh"

namespace sdgp {

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)ptr;
  }
  return fn;
}

// A tensor map is a pure function of these arguments (it holds the address, not the memory), and a training
// loop asks for the same few maps every step: each host thread keeps the last kMapCache it encoded. Outside a CUDA
// graph the four encodes of a launch otherwise cost about as much as a small layer's kernel.
struct MapKey {
  const void* base;
  uint64_t dims[5], strides[4];
  uint32_t box[5];
  int dt, rank, swz;
};
constexpr int kMapCache = 64;

}  // namespace

bool encode(CUtensorMap* tm, CUtensorMapDataType dt, int rank, const void* base, const uint64_t* dims,
            const uint64_t* strides_bytes, const uint32_t* box, CUtensorMapSwizzle swz) {
  static thread_local MapKey keys[kMapCache];
  static thread_local CUtensorMap maps[kMapCache];
  static thread_local int used = 0, next = 0;
  MapKey key;
  memset(&key, 0, sizeof(key));
  key.base = base; key.dt = (int)dt; key.rank = rank; key.swz = (int)swz;
  for (int i = 0; i < rank; ++i) { key.dims[i] = dims[i]; key.box[i] = box[i]; }
  for (int i = 0; i + 1 < rank; ++i) key.strides[i] = strides_bytes[i];
  for (int i = 0; i < used; ++i)
    if (memcmp(&keys[i], &key, sizeof(key)) == 0) {
      *tm = maps[i];
      return true;
    }
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint32_t ones[5] = {1, 1, 1, 1, 1};
  auto make = [&]() {
    return fn(tm, dt, (cuuint32_t)rank, const_cast<void*>(base), (const cuuint64_t*)dims, (const cuuint64_t*)strides_bytes,
              (const cuuint32_t*)box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  if (!make()) {
    // a thread whose first CUDA call this is has no context yet (the encoder is a driver function): cudaSetDevice binds it
    const int dev = current_device();
    if (dev < 0 || cudaSetDevice(dev) != cudaSuccess || !make()) return false;
  }
  const int slot = used < kMapCache ? used++ : (next = (next + 1) % kMapCache);
  keys[slot] = key;
  maps[slot] = *tm;
  return true;
}

namespace {

int largest_divisor_at_most(int x, int cap) {
  for (int d = cap < x ? cap : x; d >= 1; --d)
    if (x % d == 0) return d;
  return 1;
}

// Pixel patch of one 128-row tile: whole image rows when the image is narrow, so that a
// filter tap shifts the patch as a block and the image border falls outside the box.
void choose_patch(int B, int H, int W, int* TW, int* TH, int* TB) {
  if (W >= kBM) {
    *TW = kBM; *TH = 1; *TB = 1;
    return;
  }
  *TW = W;
  const int max_h = kBM / W;
  if (H <= max_h) {
    *TH = H;
    const int max_b = kBM / (W * H);
    *TB = max_b < B ? max_b : B;
    if (*TB < 1) *TB = 1;
  } else {
    const int d = largest_divisor_at_most(H, max_h);
    *TH = (2 * d >= max_h) ? d : max_h;
    *TB = 1;
  }
}

}  // namespace

// Per-device caches, indexed by the ordinal of the CURRENT device (the library follows the caller's
// current device, and a process may drive several). Filled on first use; concurrent first uses store the
// same values.
int current_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
  return dev;
}

int sm_count() {
  static int n[kMaxDevices] = {};
  const int dev = current_device();
  if (dev < 0) return 148;
  if (!n[dev]) {
    int v = 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    n[dev] = v > 0 ? v : 148;
  }
  return n[dev];
}

namespace {

// Channel blocks of dL/dO (kbc channels each, `all` in total) a tile of `bn` input channels has to visit: all of them, or, with
// a block-diagonal W, the widest window of blocks any tile needs.
int k_window(int bn, int channels, int all, int kbc, int Cout, const ConvGroups* groups) {
  if (!groups || groups->cin_g <= 0 || groups->cout_g <= 0) return all;
  int widest = 0;
  for (int n0 = 0; n0 < channels; n0 += bn) {
    const int lo = (n0 / groups->cin_g) * groups->cout_g / kbc;
    int co_end = ((n0 + bn + groups->cin_g - 1) / groups->cin_g) * groups->cout_g;
    if (co_end > Cout) co_end = Cout;
    const int hi = (co_end + kbc - 1) / kbc;
    if (hi - lo > widest) widest = hi - lo;
  }
  return widest > 0 && widest < all ? widest : all;
}

// Input channels per tile of the general kernel. A tile's main loop is bound by the bytes an SM pulls in from L2 per channel block (16 KB of A, and
// W in proportion to BN) and it has a fixed part, so a round of tiles costs about k_blocks * (256 + 2 BN) + 256 units; the last tile
// of a row may be partly empty (columns past the stored channels are computed and not stored). Narrow tiles win where there
// are too few for every CTA pair (1777 x 1088 . 1088 x 832: 14.7 -> 10.9 us), 192 where 128 or 256 would leave a third of the columns
// idle or double the tiles (10736 x 1152 . 1152 x 576: 31 -> 19 us, prune included).
int choose_bn(int64_t m_tiles, int channels, int all, int kbc, int Cout, const ConvGroups* groups) {
  const int64_t pairs = sm_count() / 2, rows = (m_tiles + 1) / 2;
  int best = 64;
  int64_t best_cost = INT64_MAX;
  for (int bn = 64; bn <= 256; bn += 64) {
    const int64_t tiles = rows * ((channels + bn - 1) / bn);
    const int64_t cost = (tiles + pairs - 1) / pairs * (256 + k_window(bn, channels, all, kbc, Cout, groups) * (256 + 2 * bn));
    if (cost <= best_cost) { best = bn; best_cost = cost; }
  }
  return best;
}

// Whole-filter reuse pays when there is more than one tap and strips of 8 x 16 pixels (images at most 8 pixels tall: 8 rows of two
// images) cover the image without too much padding. How much is too much was measured (two-pass, us, general kernel -> this one): nine
// taps, 27 x 27 (140 % covered) 34.5 -> 16.8, 13 x 13 (151 %) 49 -> 27.5, 10 x 10 (256 %) 18.6 -> 15.8, 9 x 9 (316 %) 15.6 -> 19.3;
// two to four taps, 7 x 7 (131 %) 31 -> 37. Pruning inside the general kernel costs so much more that the fused mode takes
// any image of at least 5 x 5 (9 x 9: 36.7 -> 24.5).
bool halo_applies(int H, int W, int taps, bool sparse, bool fused) {
  if (taps < 2) return false;
  // two images per strip row, four pixel rows of eight images per strip. With a sparse A only: fused, it prunes each box S times instead
  // of R * S times; two-pass it measured the same as the general kernel; the dense twin measured slower there (one tile per CTA
  // pair: set-up and the single epilogue dominate either way).
  if (W == 4 && H >= 3 && H <= 4) return sparse;
  if (W < 5 || H < 5) return false;
  if (fused) return true;
  if (taps < 6 && (W < 8 || (H < 12 && H > 8) || H < 6)) return false;
  const int th = H <= 8 ? 8 : kHaloRows;
  const int64_t covered = (int64_t)((W + 7) / 8 * 8) * ((H + th - 1) / th * th);
  return covered * 100 <= (int64_t)H * W * (taps < 6 ? 135 : 260);
}

// Estimated time of one launch of that kernel over bn input channels and nt strips per tile, in units of the fixed part of a tap (some
// 0.3 us: barriers and the MMA issue, whatever the width). A round of tiles takes, per channel block, its taps at 1 + 1/8 per 64
// accumulator columns (dense A: 1/16) and the box's bytes or - fused - the pruning of the box, whichever is longer; then an epilogue. Two
// strips side by side share every W stage and the fixed part; where there are too few strips for every CTA pair, or a box's pruning
// sets the pace, one is better. Constants fitted to 790 layers timed in all six shapes, dense, two-pass and fused: 0.3 % behind the best
// shape in the mean, more than 5 % behind in 20 of them. A rule that looked at the width alone was 2.4 % behind. Us, that rule and this one:
// 20 x 4 x 4 images, 256 -> 256, fused, random 2:16, 49.6, 30.5; 110 x 32 x 32, 256 -> 384, dense after pruning, 169.8, 139.3; 339 x 14 x 14,
// 12 groups of 16, 53.7, 39.7; 32 x 28 x 28, 128 -> 320, 11 x 11, fused (192 columns do not fit), 1034, 265. 0: no such shape for this layer.
double halo_cost(int B, int H, int W, int R, int S, int bn, int nt, bool sparse, int tiles_n, int k_blocks, const FusedPrune* fused) {
  const bool split = W == 4;
  if (nt * bn > 256 || (!split && nt == 2 && W <= 8)) return 0.0;
  const int per_row = split ? 2 * nt : 1, th = H <= 4 ? 4 : H <= 8 ? 8 : kHaloRows, tb = kHaloRows / th;
  if (B % per_row != 0) return 0.0;
  const int sb = split ? 1 : S, boxes = split ? S : 1;
  const int sets_w = split ? 1 : (W + 8 * nt - 1) / (8 * nt), tiles_h = (H + th - 1) / th;
  const int64_t sets = (int64_t)sets_w * tiles_h * ((B + tb * per_row - 1) / (tb * per_row));
  const int64_t pairs = sm_count() / 2, rounds = ((sets + 1) / 2 * tiles_n + pairs - 1) / pairs;
  const double columns = nt * bn / 64.0, img_rows = (8 * nt + sb - 1) * (th + R - 1) * tb;
  double box = R * sb * (1.0 + columns * (sparse ? 0.125 : 0.0625)) + 0.003 * img_rows;
  if (fused) {
    const bool whole_images = sets_w == 1 && tiles_h == 1;  // only the units inside the images are pruned (plan_halo())
    const double units = whole_images ? (H < th ? H : th) * tb * nt : img_rows / 8;
    const double unit = fused->scheme == SDGP_MAGNITUDE ? 0.37 : fused->scheme == SDGP_RANDOM ? 0.92 : 1.1;
    if (5.0 + units * unit > box) box = 5.0 + units * unit;
  }
  return (double)rounds * (k_blocks * boxes * box + 4.3 + 0.5 * columns);
}

// The same for the four output parities of a stride-2 convolution in one launch, the mean over them per unit; H, W: their largest images,
// R, S: the whole filter. A unit's stores take at least 2.2 per 64 columns (they are what bounds parities of one or two taps).
double halo_cost_classes(int B, int H, int W, int R, int S, int pad, int bn, int nt, bool sparse, int tiles_n, int k_blocks) {
  if (nt * bn > 256 || (nt == 2 && W <= 8)) return 0.0;
  const int th = H <= 8 ? 8 : kHaloRows, tb = kHaloRows / th;
  const int sets_w = (W + 8 * nt - 1) / (8 * nt), tiles_h = (H + th - 1) / th;
  const int64_t sets = (int64_t)sets_w * tiles_h * ((B + tb - 1) / tb);
  const int64_t pairs = sm_count() / 2, rounds = ((sets + 1) / 2 * tiles_n * 4 + pairs - 1) / pairs;
  const double columns = nt * bn / 64.0, img_rows = (8 * nt + (S + 1) / 2 - 1) * (th + (R + 1) / 2 - 1) * tb;
  double sum = 0.0;
  for (int c = 0; c < 4; ++c) {
    const int Rc = (R - ((c >> 1) + pad) % 2 + 1) / 2, Sc = (S - ((c & 1) + pad) % 2 + 1) / 2;
    const double box = Rc * Sc * (1.0 + columns * (sparse ? 0.125 : 0.0625)) + 0.003 * img_rows;
    const double main_loop = k_blocks * box, stores = 2.2 * columns;
    sum += (main_loop > stores ? main_loop : stores) + 4.3 + 0.5 * columns;
  }
  return (double)rounds * sum / 4.0;
}

// Whether one launch for the four parities is faster than one each. It saves three launches and reads of dL/dO, some 25 us, but its strips
// are laid out for the largest parity's images, where the general kernel's patches, which most classes of small images get otherwise, fit
// each parity's (some 125 %); and with a dense A the general kernel is the faster one per product. The constants (us per 1e9 products, one
// launch and four) follow 34 layers timed both ways. Us, four launches -> one, prune kernel included, sparse: 265 x 13 x 13 images, 896 -> 896
// (160 % covered) 122 -> 156; 60 x 20 x 20, 512 -> 512 (256 %) 41 -> 48; 325 x 27 x 27, 128 -> 128 54 -> 34; 479 x 14 x 14, 448 -> 256 68 -> 49;
// 18 x 32 x 32, 384 -> 128 25 -> 10. Dense after pruning: 64 x 27 x 27, 896 -> 896 212 -> 264; 256 x 16 x 16, 512 -> 512 (100 %) 100 -> 83.
bool classes_pay(int B, int H, int W, int Cin, int Cout, int R, int S, int pad, bool sparse) {
  const int H0 = (H + 1) / 2, W0 = (W + 1) / 2, th = H0 <= 8 ? 8 : kHaloRows;
  const double covered = (double)((W0 + 7) / 8 * 8) * ((H0 + th - 1) / th * th);
  double one = 0.0, four = 0.0;  // positions times taps
  for (int c = 0; c < 4; ++c) {
    const int ph = c >> 1, pw = c & 1, taps = ((R - (ph + pad) % 2 + 1) / 2) * ((S - (pw + pad) % 2 + 1) / 2);
    one += taps * covered;
    four += (double)taps * ((H - ph + 1) / 2) * ((W - pw + 1) / 2);
  }
  const double excess = sparse ? 0.87 * one - 1.09 * four : 1.05 * one - 0.96 * four;
  return 2.0e-9 * excess * B * Cin * Cout < (sparse ? 25.0 : 20.0);
}

// A tile of the strip kernel: input channels, strips side by side, estimated time.
struct TileShape {
  int bn, nt;
  double cost;
};

// Channel blocks that a tile of bn input channels visits (grouped convolutions: a window of them).
void set_width(HaloParams* p, int bn, int channels, int kb_channels, const ConvGroups* groups) {
  const int blocks = (p->Cout + kb_channels - 1) / kb_channels;
  p->tiles_n = (channels + bn - 1) / bn;
  p->k_blocks = k_window(bn, channels, blocks, kb_channels, p->Cout, groups);
  p->diag_cin_g = p->diag_cout_g = p->diag_last = 0;
  if (p->k_blocks < blocks) {
    p->diag_cin_g = groups->cin_g; p->diag_cout_g = groups->cout_g;
    p->diag_last = blocks - p->k_blocks;
  }
}

// All four output parities of a strided layer in one launch of the strip kernel, where its strips cover their images well enough (the
// same bounds as for a filter of its size at stride 1) and that is estimated to be faster: its parameters and the tile shapes, cheapest first.
bool plan_parities(bool sparse, const DgradView& view, int B, int H, int W, int Cin, int Cout, int R, int S, int stride, int pad,
                   const ConvGroups* conv_groups, HaloParams* hp, TileShape (&shapes)[6]) {
  if (stride != 2 || R < 2 || S < 2 || W <= 8 || !halo_applies((H + 1) / 2, (W + 1) / 2, R * S, sparse, false) ||
      !classes_pay(B, H, W, view.d.channels, view.a_channels, R, S, pad, sparse))
    return false;
  *hp = HaloParams{};
  hp->B = B; hp->H = (H + 1) / 2; hp->W = (W + 1) / 2; hp->Cin = Cin; hp->Cout = Cout;
  hp->r_step = hp->s_step = 2;
  hp->S_full = S;
  hp->P = view.P; hp->Q = view.Q;
  hp->last_launch = 1;
  hp->classes = 4;
  for (int c = 0; c < 4; ++c) {
    HaloClass& k = hp->cls[c];
    const int ph = c >> 1, pw = c & 1;
    k.r_first = (ph + pad) % 2; k.s_first = (pw + pad) % 2;
    k.R = (R - k.r_first + 1) / 2; k.S = (S - k.s_first + 1) / 2;
    k.pad_h = (ph + pad - k.r_first) / 2; k.pad_w = (pw + pad - k.s_first) / 2;
    k.H = (H - ph + 1) / 2; k.W = (W - pw + 1) / 2;
    hp->R = k.R > hp->R ? k.R : hp->R;
    hp->S = k.S > hp->S ? k.S : hp->S;
  }
  const int kb_channels = sparse ? 128 : 64, blocks = (Cout + kb_channels - 1) / kb_channels;
  hp->k_last = blocks - 1;
  const int left = view.a_channels - hp->k_last * kb_channels, per_mma = kb_channels / 4;
  hp->last_mmas = left < kb_channels ? (left + per_mma - 1) / per_mma : 4;
  const TileShape all[] = {{64, 1, 0}, {64, 2, 0}, {128, 1, 0}, {128, 2, 0}, {192, 1, 0}, {256, 1, 0}};
  for (int i = 0; i < 6; ++i) {
    shapes[i] = all[i];
    set_width(hp, all[i].bn, view.d.channels, kb_channels, conv_groups);
    const double cost = halo_cost_classes(B, hp->H, hp->W, R, S, pad, all[i].bn, all[i].nt, sparse, hp->tiles_n, hp->k_blocks);
    shapes[i].cost = cost > 0.0 ? cost : 1e9;
  }
  std::sort(std::begin(shapes), std::end(shapes), [](const TileShape& a, const TileShape& b) { return a.cost < b.cost; });
  return true;
}

// What a call reads and writes per pixel; base and strides of dD are the launch's.
DgradView dgrad_view(int B, int H, int W, int Cin, int Cout, int R, int S, int stride, int pad, const StoredChannels* stored) {
  DgradView view = {};
  view.P = (H + 2 * pad - R) / stride + 1;
  view.Q = (W + 2 * pad - S) / stride + 1;
  view.batch = B;
  view.a_channels = (stored && stored->a) ? stored->a : Cout;
  view.meta_channels = (view.a_channels + 127) / 128 * 128;
  view.d.channels = (stored && stored->d) ? stored->d : Cin;
  view.w_cols = (int64_t)R * S * Cin;
  return view;
}

// What pruning costs (measured on a [16384 x 4096] tensor and on 50176 x 1024 rows): clocks of the rows kernel's pruning warps per block of
// 128 channels, picoseconds per element of the prune kernel where the integer pipe bounds it.
struct PruneCost {
  int stage_clk;
  double ps;
};
PruneCost prune_cost(int m, int scheme) {
  if (scheme == SDGP_RANDOM) return m == 4 ? PruneCost{3600, 0.68} : PruneCost{4300, 0.90};
  if (scheme == SDGP_RESCALED_MAGNITUDE) return m == 4 ? PruneCost{3100, 0.56} : PruneCost{3800, 0.69};
  return m == 4 ? PruneCost{1700, 0.40} : PruneCost{2500, 0.57};
}

}  // namespace

// A: dense dL/dO [B,P,Q,Cout] (sparse == false) or compressed values [B,P,Q,Cout/2] with meta [B,P,Q,Cp/16], Cp = Cout
// rounded up to 128 (pad channels name the position pair (0,1)); Wt: [Cout, R, S, Cin]; dD: [B,H,W,Cin].
// Stride 2 is split by the parity of the output pixel: pixel (2h'+ph, 2w'+pw) only meets the taps
// r = ph + pad (mod 2), s = pw + pad (mod 2), and on those it is a stride-1 problem from dO to
// the strided view dD[:, ph::2, pw::2, :].
// fused != nullptr (with sparse == true): A is the DENSE dL/dO and the kernel prunes it itself (n = 1 or 2; m = 4, 8 or 16, in the
// strip kernel also 32); no compressed tensor exists in global memory.
sdgp_status launch_dgrad(bool sparse, const void* A, const void* meta, const void* Wt, void* dD, int B,
                         int H, int W, int Cin, int Cout, int R, int S, int stride, int pad, cudaStream_t stream,
                         const FusedPrune* fused, int dtype, const StoredChannels* stored, const ConvGroups* conv_groups) {
  if (fused && stored) return SDGP_ERR_UNSUPPORTED;  // the pruning warps address dL/dO by the channel count they tile by
  if (stored && (stored->a < 0 || stored->a > Cout || stored->a % 8 != 0 || stored->d < 0 || stored->d > Cin || stored->d % 8 != 0))
    return SDGP_ERR_INVALID_ARG;
  if (fused && (!sparse || fused->n < 1 || fused->n > 2)) return SDGP_ERR_UNSUPPORTED;
  if (fused && fused->m != 4 && fused->m != 8 && fused->m != 16 && fused->m != 32) return SDGP_ERR_UNSUPPORTED;
  if (dtype != SDGP_BF16 && dtype != SDGP_FP16) return SDGP_ERR_INVALID_ARG;
  if (fused && dtype == SDGP_FP16 && fused->scheme == SDGP_RESCALED_MAGNITUDE) return SDGP_ERR_UNSUPPORTED;
  if (stride != 1 && stride != 2) return SDGP_ERR_UNSUPPORTED;
  if (R == 1 && S == 1 && stride == 1 && pad == 0 && (int64_t)B * H * W <= 0x7FFFFFFF) {
    // a 1 x 1 convolution is a fully connected layer over its pixels: tiles of 128 of them whatever the image size
    W = B * H * W;
    B = H = W > 0 ? 1 : 0;
  }
  if ((int64_t)B * H * W == 0) return SDGP_OK;
  const int P = (H + 2 * pad - R) / stride + 1, Q = (W + 2 * pad - S) / stride + 1;
  if (P < 1 || Q < 1) return SDGP_ERR_INVALID_ARG;
  if (Cin % 64 != 0 || Cout % 64 != 0) return SDGP_ERR_UNSUPPORTED;
  if ((int64_t)R * S * Cin > 0x7FFFFFFF) return SDGP_ERR_UNSUPPORTED;

  if (fused && B == 1 && H == 1 && R == 1 && S == 1 && stride == 1 && pad == 0 && fused->m <= 16) {
    const RowsPlan plan = plan_rows(W, Cout, Cin, prune_cost(fused->m, fused->scheme).stage_clk);
    // The rows kernel's warps prune 8 rows each of all 128, whatever exists; the general kernel's 384 pruning threads an eighth of a row each,
    // 48 rows in one pass. Where pruning sets the pace (random and rescaled functions) few rows are faster there: 35 x 3264 . 3264 x 192,
    // random 2:16, 48.4 us against 68.7; 36 x 896 . 896 x 576, rescaled 1:4, 14.2 against 15.3; magnitude 47 x 2944 . 2944 x 64 35.4 against 33.9.
    const bool few_rows = W <= 48 && fused->scheme != SDGP_MAGNITUDE;
    if (plan.ok && !few_rows) return launch_rows_fused(plan, A, Wt, Cout, Cin, dD, *fused, dtype, stream);
  }
  const int kb_channels = sparse ? 128 : 64;

  DgradView view = dgrad_view(B, H, W, Cin, Cout, R, S, stride, pad, stored);
  const size_t Cd = (size_t)view.d.channels;

  HaloParams hp4;
  TileShape shapes4[6];
  if (!fused && plan_parities(sparse, view, B, H, W, Cin, Cout, R, S, stride, pad, conv_groups, &hp4, shapes4)) {
    hp4.f16 = dtype == SDGP_FP16 ? 1 : 0;
    view.d.base = (uint8_t*)dD;
    view.d.sw = 2 * (int64_t)Cd * 2;
    view.d.sh = 2 * (int64_t)W * Cd * 2;
    view.d.sb = (int64_t)H * W * Cd * 2;
    view.d.aligned32 = 0;
    for (const TileShape& s : shapes4) {
      set_width(&hp4, s.bn, view.d.channels, kb_channels, conv_groups);
      const sdgp_status st = sparse ? launch_halo_sparse(s.bn, s.nt, A, meta, Wt, view, hp4, stream) : launch_halo_dense(s.bn, s.nt, A, Wt, view, hp4, stream);
      if (st != SDGP_ERR_UNSUPPORTED) return st;
    }
  }

  // Output parities that no tap reaches are zero: clear dD first if there is any such class.
  bool any_empty = false;
  int last_class = 0;  // of those that launch a kernel
  const int all_blocks = (Cout + kb_channels - 1) / kb_channels;
  // Tile shapes of the strip kernel, one for all classes of the call (kernels that alternate between shapes measured up to 10 % slower).
  TileShape shapes[] = {{64, 1, 0}, {64, 2, 0}, {128, 1, 0}, {128, 2, 0}, {192, 1, 0}, {256, 1, 0}};
  for (int ph = 0; ph < stride; ++ph)
    for (int pw = 0; pw < stride; ++pw) {
      const int r0 = (ph + pad) % stride, s0 = (pw + pad) % stride;
      if (r0 >= R || s0 >= S) { any_empty = true; continue; }
      if (ph >= H || pw >= W) continue;
      last_class = ph * stride + pw;
      const int Hs = (H - ph + stride - 1) / stride, Ws = (W - pw + stride - 1) / stride;
      const int Rs = (R - r0 + stride - 1) / stride, Ss = (S - s0 + stride - 1) / stride;
      if (!halo_applies(Hs, Ws, Rs * Ss, sparse, fused != nullptr)) continue;
      for (TileShape& s : shapes) {
        const int tiles_n = (view.d.channels + s.bn - 1) / s.bn;
        const double cost = halo_cost(B, Hs, Ws, Rs, Ss, s.bn, s.nt, sparse, tiles_n,
                                      k_window(s.bn, view.d.channels, all_blocks, kb_channels, Cout, conv_groups), fused);
        s.cost += cost > 0.0 ? cost : 1e9;  // (does not exist for this class: tried last)
      }
    }
  std::sort(std::begin(shapes), std::end(shapes), [](const TileShape& a, const TileShape& b) { return a.cost < b.cost; });
  if (any_empty && cudaMemsetAsync(dD, 0, (size_t)B * H * W * Cd * 2, stream) != cudaSuccess) return SDGP_ERR_CUDA;
  for (int ph = 0; ph < stride; ++ph) {
    for (int pw = 0; pw < stride; ++pw) {
      const int Hs = (H - ph + stride - 1) / stride, Ws = (W - pw + stride - 1) / stride;  // pixels of this class
      if (Hs <= 0 || Ws <= 0) continue;
      DgradParams p = {};
      p.r_first = (ph + pad) % stride; p.r_step = stride;
      p.s_first = (pw + pad) % stride; p.s_step = stride;
      p.S_full = S;
      p.R = p.r_first < R ? (R - p.r_first + stride - 1) / stride : 0;
      p.S = p.s_first < S ? (S - p.s_first + stride - 1) / stride : 0;
      if (p.R == 0 || p.S == 0) continue;  // cleared above
      p.pad_h = (ph + pad - p.r_first) / stride;
      p.pad_w = (pw + pad - p.s_first) / stride;
      p.B = B; p.H = Hs; p.W = Ws; p.Cin = Cin; p.Cout = Cout;
      choose_patch(B, Hs, Ws, &p.TW, &p.TH, &p.TB);
      p.tiles_w = (Ws + p.TW - 1) / p.TW;
      p.tiles_h = (Hs + p.TH - 1) / p.TH;
      p.tiles_b = (B + p.TB - 1) / p.TB;
      const int64_t m_tiles = (int64_t)p.tiles_w * p.tiles_h * p.tiles_b;
      p.m_tiles = (int)m_tiles;
      // what depends on the width of a tile
      auto set_width = [&](int bn) {
        p.tiles_n = (view.d.channels + bn - 1) / bn;
        p.k_blocks = k_window(bn, view.d.channels, all_blocks, kb_channels, Cout, conv_groups);
        p.diag_cin_g = p.diag_cout_g = p.diag_last = 0;
        if (p.k_blocks < all_blocks) {
          p.diag_cin_g = conv_groups->cin_g; p.diag_cout_g = conv_groups->cout_g;
          p.diag_last = all_blocks - p.k_blocks;
        }
      };
      // the last channel block may be partly empty: its MMAs (32 channels each, dense 16) past the channels that exist are left out
      p.k_last = all_blocks - 1;
      const int left = view.a_channels - p.k_last * kb_channels, per_mma = kb_channels / 4;
      p.last_mmas = left < kb_channels ? (left + per_mma - 1) / per_mma : 4;
      p.P = P; p.Q = Q;
      p.f16 = dtype == SDGP_FP16 ? 1 : 0;
      p.last_launch = ph * stride + pw == last_class;
      if (fused) {
        p.fused_n = fused->n; p.fused_m = fused->m; p.fused_scheme = fused->scheme;
        p.seed_lo = (uint32_t)fused->seed; p.seed_hi = (uint32_t)(fused->seed >> 32);
      }
      view.d.base = (uint8_t*)dD + ((size_t)ph * W + pw) * Cd * 2;
      view.d.sw = (int64_t)stride * Cd * 2;
      view.d.sh = (int64_t)stride * W * Cd * 2;
      view.d.sb = (int64_t)H * W * Cd * 2;
      view.d.aligned32 = ((uintptr_t)dD & 31u) == 0 && Cd % 16 == 0;
      sdgp_status st = SDGP_ERR_UNSUPPORTED;
      if (halo_applies(Hs, Ws, p.R * p.S, sparse, fused != nullptr)) {
        HaloParams hp = {};
        hp.classes = 1;
        hp.B = B; hp.H = Hs; hp.W = Ws; hp.Cin = Cin; hp.Cout = Cout;
        hp.R = p.R; hp.S = p.S; hp.pad_h = p.pad_h; hp.pad_w = p.pad_w;
        hp.r_first = p.r_first; hp.r_step = p.r_step; hp.s_first = p.s_first; hp.s_step = p.s_step;
        hp.S_full = S;
        hp.P = P; hp.Q = Q;
        hp.k_last = p.k_last; hp.last_mmas = p.last_mmas;
        hp.f16 = p.f16;
        hp.last_launch = p.last_launch;
        if (fused) {
          hp.fused_n = p.fused_n; hp.fused_m = p.fused_m; hp.fused_scheme = p.fused_scheme; hp.seed_lo = p.seed_lo; hp.seed_hi = p.seed_hi;
        }
        // from the cheapest on, until one fits shared memory (a large filter's box and a wide tile may not)
        for (const TileShape& s : shapes) {
          set_width(s.bn);
          hp.tiles_n = p.tiles_n; hp.k_blocks = p.k_blocks;
          hp.diag_cin_g = p.diag_cin_g; hp.diag_cout_g = p.diag_cout_g; hp.diag_last = p.diag_last;
          st = fused    ? launch_halo_fused(s.bn, s.nt, A, Wt, view, hp, stream)
               : sparse ? launch_halo_sparse(s.bn, s.nt, A, meta, Wt, view, hp, stream)
                        : launch_halo_dense(s.bn, s.nt, A, Wt, view, hp, stream);
          if (st != SDGP_ERR_UNSUPPORTED) break;
        }
        if (st == SDGP_OK) continue;
        if (st != SDGP_ERR_UNSUPPORTED) return st;  // otherwise: no shape fits, use the general kernel
      }
      if (fused && fused->m == 32) return SDGP_ERR_UNSUPPORTED;  // this kernel's threads hold 16 channels each: groups of up to 16
      const int BN = choose_bn(m_tiles, view.d.channels, all_blocks, kb_channels, Cout, conv_groups);
      set_width(BN);
      if (m_tiles * p.tiles_n > 0x3FFFFFFF) return SDGP_ERR_UNSUPPORTED;
      p.pair_tiles = (int)((m_tiles + 1) / 2) * p.tiles_n;
      st = launch_general(sparse, fused != nullptr, BN, A, meta, Wt, view, p, stream);
      if (st != SDGP_OK) return st;
    }
  }
  return SDGP_OK;
}

namespace {

// Two-pass calls over rows: the kernel that prunes inside the contraction replaces prune kernel + contraction where it is
// estimated to be faster. Estimate of the pair, us: 4 for two launches' ramps, the prune kernel's bytes at 6.4 TB/s or its
// arithmetic, and the contraction's bytes, operand traffic from L2 or products; of the one kernel, 0.8 of plan_rows()'s clocks. Few channels
// (one launch less, no second read of dO) favour the rows kernel, many channels on few rows the pair (a CTA pair prunes its blocks one after
// another). Of 1540 drawn layers timed both ways the estimate picks a kernel more than 5 % behind the other on 76, more than 10 % on 31, 0.6 % in
// the mean; with 5.5 and 0.9, from when the pair was slower, 140, 73 and 1.2 %.
bool rows_fused_pays(int64_t rows, int K, int N, int m, int scheme, RowsPlan* plan) {
  const PruneCost pc = prune_cost(m, scheme);
  *plan = plan_rows(rows, K, N, pc.stage_clk);
  if (!plan->ok) return false;
  const double e = (double)rows * K, out = (double)rows * N;
  const double prune_mem = 3.125 * e / 6.4e6, prune_alu = e * pc.ps * 1e-6, prune = prune_mem > prune_alu ? prune_mem : prune_alu;
  const int64_t m_tiles = (rows + 127) / 128;
  const int blocks = (K + 127) / 128, bn = choose_bn(m_tiles, N, blocks, 128, K, nullptr);
  const int64_t tiles = (m_tiles + 1) / 2 * ((N + bn - 1) / bn), pairs = sm_count() / 2;
  const double l2 = (double)((tiles + pairs - 1) / pairs) * (256 + blocks * (256 + 2 * bn)) / 1900.0;
  const double mem = (1.125 * e + 2.0 * out) / 6.0e6, mma = 2.0 * e * N / 2.0e9;
  double contraction = mem > l2 ? mem : l2;
  if (mma > contraction) contraction = mma;
  return plan->cost / 1900.0 * 0.8 < 4.0 + prune + contraction;
}

}  // namespace

// Prune kernel, block-diagonal filters and contraction of a grouped layer. Constants fitted to the same layers as estimate_grouped()'s: within 9 % for
// nine in ten of 1088 others.
double estimate_block_diagonal(int B, int H, int W, int C, int groups, int R, int S, int pad, const FusedPrune& prune) {
  const int P = H + 2 * pad - R + 1, Q = W + 2 * pad - S + 1, Ck = (C + 63) / 64 * 64, blocks = (Ck + 127) / 128;
  const ConvGroups cg = {C / groups, C / groups};
  const double e = (double)B * P * Q * C, filters = 2.0 * Ck * R * S * Ck;
  const double prune_mem = 3.125 * e / 6.4e6, prune_alu = e * prune_cost(prune.m, prune.scheme).ps * 1e-6;
  const double before = 6.7 + 1.37 * (prune_mem > prune_alu ? prune_mem : prune_alu) + 0.25e-6 * filters;
  if (halo_applies(H, W, R * S, true, false)) {
    double best = 0.0;
    const TileShape all[] = {{64, 1, 0}, {64, 2, 0}, {128, 1, 0}, {128, 2, 0}, {192, 1, 0}, {256, 1, 0}};
    for (const TileShape& s : all) {
      const double cost = halo_cost(B, H, W, R, S, s.bn, s.nt, true, (C + s.bn - 1) / s.bn, k_window(s.bn, C, blocks, 128, Ck, &cg), nullptr);
      if (cost > 0.0 && (best == 0.0 || cost < best)) best = cost;
    }
    if (best > 0.0) return before + 0.187 * best;
  }
  int64_t m_tiles;
  if (R == 1 && S == 1 && pad == 0) {
    m_tiles = ((int64_t)B * H * W + kBM - 1) / kBM;
  } else {
    int TW, TH, TB;
    choose_patch(B, H, W, &TW, &TH, &TB);
    m_tiles = (int64_t)((W + TW - 1) / TW) * ((H + TH - 1) / TH) * ((B + TB - 1) / TB);
  }
  const int bn = choose_bn(m_tiles, C, blocks, 128, Ck, &cg);
  const int64_t tiles = (m_tiles + 1) / 2 * ((C + bn - 1) / bn), pairs = sm_count() / 2;
  return before + 0.5 + 1.8 * (double)((tiles + pairs - 1) / pairs) * (256.0 + (double)k_window(bn, C, blocks, 128, Ck, &cg) * R * S * (256 + 2 * bn)) / 1900.0;
}

bool query_parities(bool sparse, int B, int H, int W, int Cin, int Cout, int R, int S, int stride, int pad, const StoredChannels* stored,
                    const ConvGroups* conv_groups, int* plan) {
  const DgradView view = dgrad_view(B, H, W, Cin, Cout, R, S, stride, pad, stored);
  HaloParams hp;
  TileShape shapes[6];
  if (!plan_parities(sparse, view, B, H, W, Cin, Cout, R, S, stride, pad, conv_groups, &hp, shapes)) return false;
  for (const TileShape& s : shapes) {
    set_width(&hp, s.bn, view.d.channels, sparse ? 128 : 64, conv_groups);
    HaloParams p = hp;
    if (!(sparse ? plan_halo_sparse(s.bn, s.nt, &p) : plan_halo_dense(s.bn, s.nt, &p))) continue;
    plan[0] = 2; plan[1] = p.units; plan[2] = p.split_from; plan[3] = pairs_for(p.units); plan[4] = s.bn; plan[5] = s.nt; plan[6] = p.tb;
    return true;
  }
  return false;
}

sdgp_status try_rows_fused(const void* dO, const void* W, void* dD, int64_t rows, int K, int N, const FusedPrune& prune, int dtype,
                           cudaStream_t stream, bool* taken) {
  RowsPlan plan;
  *taken = rows_fused_pays(rows, K, N, prune.m, prune.scheme, &plan);
  return *taken ? launch_rows_fused(plan, dO, W, K, N, dD, prune, dtype, stream) : SDGP_OK;
}

// One CTA waits, with a 50 ms limit, on a barrier that nothing ever signals: the wait must give
// up, record its code and let the kernel end normally.
__global__ void bounded_wait_selftest_kernel() {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    ptx::mbar_init(&bar, 1);
    ptx::fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) ptx::mbar_wait(&bar, 0u, &g_device_error, 0xE00u, 50000000ull);
  __syncthreads();
}

sdgp_status launch_bounded_wait_selftest(cudaStream_t stream) {
  bounded_wait_selftest_kernel<<<1, 32, 0, stream>>>();
  return cudaGetLastError() == cudaSuccess ? SDGP_OK : SDGP_ERR_CUDA;
}

sdgp_status read_device_error() {
  if (cudaDeviceSynchronize() != cudaSuccess) return SDGP_ERR_CUDA;
  bool timed_out = false;
  cudaError_t (*const words[])(unsigned int*) = {take_error_word, take_error_general, take_error_halo_sparse, take_error_halo_dense,
                                                 take_error_halo_fused, take_error_rows, take_error_grouped};
  for (auto take : words) {
    unsigned int word = 0;
    if (take(&word) != cudaSuccess) return SDGP_ERR_CUDA;
    timed_out |= word != 0;
  }
  return timed_out ? SDGP_ERR_TIMEOUT : SDGP_OK;
}

}  // namespace sdgp
