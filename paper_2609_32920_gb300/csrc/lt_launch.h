// lt_launch.h -- internal interface between the C-ABI host code and the kernels.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace lt {

struct DevScene;

// Primitives of a path's first vertices as kept in its per-path record: `bits` each (enough for
// the scene's primitives), at most `cap` of them for a path with several valid connections and
// `cap1` for one with one (160 and 96 bits, and 32 more where the validity bits need one word).
// `one`: a path with one valid connection has that connection in its record (and not
// delta_total); see lrb3_state_bytes.
struct HitBits {
  int bits, cap, cap1, one;
};
// Paths of at most 32 vertices need one word of validity bits; their second one holds hits.
__host__ __device__ inline bool one_mask_word(int max_depth) { return max_depth <= 32; }

// Per-call kernel parameters (by value).
struct KParams {
  uint64_t seed;
  int64_t path_offset;
  int64_t n_paths;
  int max_depth;
  float inv_n;               // 1 / N of the estimator
  const float* Le;           // DEVICE [3]
  const float* albedo;       // DEVICE [n_albedo]
  const uint8_t* mask;       // DEVICE [n_paths] or null
  uint32_t* hash;            // DEVICE [n_paths] or null
  float* dbg;                // DEVICE [n_paths][4] or null
  size_t tape_offset;        // naive tape: bytes before the first record
  unsigned long long* census;  // DEVICE [5] or null: rays, box tests, primitive tests, vertices, connections
  int n_alb, n_h;              // albedo / height gradients accumulated in shared memory per block
                               // (array lengths, or 0: that array goes to global memory directly)
  int priv_n;                  // n_alb + n_h: floats of dynamic shared memory per block
  const float* mlp;            // learned reservoir target parameters (DEVICE) or null (luminance)
  uint32_t* order;             // plain primal: the order in which it takes the paths (or null)
  unsigned long long* order_n; // and how many are in it (the others ended on their first ray)
  void* vstate;                // plain primal: LRB-3 per-path state that receives each path's
                               // connection-validity mask (or null)
  int rr_depth;                // Russian roulette after vertices of depth >= rr_depth (0: off)
  float rr_q;                  // survival probability of the roulette
  int filter;                  // reconstruction filter: 0 tent, 1 truncated Gaussian
  uint32_t* list;              // paths with a valid connection (plain primal: appends;
                               // LRB-3 passes 2 and 3 with known masks: visit only these) or null
  unsigned long long* list_n;  // length of `list`
  unsigned long long* ticket;  // zeroed counters of entries taken: [0] pass 2, [1] pass 3 (plain
                               // primal with the LRB-3 state: [0] its 32-path chunks)
  uint32_t* multi;             // LRB-3 backward with a list: its paths with several connections
  unsigned long long* multi_n; // (k_lrb3_several appends, pass 2 visits), and their number
  double* le_sum;              // zeroed: the passes' block sums of the emitted-radiance gradient (3), and
                               // after them the blocks of pass 3 that are done (uint64); or null
  HitBits hits;                // primitives kept in the per-path records (bits 0: none)
  float4* rep;                 // LRB-3 pass 3: copies of the albedo gradient, [material][2^rep_bits]
  int rep_bits;                // (see scatter_albedo_rep), or null
  int jac_noise;               // paper-literal transport: Jacobian noise at diffuse vertices
  uint64_t noise_seed;         // its Philox key
  float det_eps;               // its determinant guard
};

struct GradPtrs {
  float* d_albedo;
  float* d_Le;
  float* d_heights;
};

struct LaunchCfg {
  int block;
  int blocks_per_sm;
  int sms;
};

struct RefitArgs {
  float4* prim;
  const int4* prim_h;
  const float4* tri_base;
  const float* heights;
  int n_prims;
  float4* node;
  const int2* range;
  int n_nodes;
  const int* big;  // nodes whose primitive range exceeds kRefitBig: a whole block reduces each
  int n_big;
  // wide BVHs (width 4 and 8): child slot -> binary node whose box it takes (-1: empty)
  float4* wnode[2];
  const int* wmap[2];
  int n_wnodes[2];
};

// Binary BVH nodes with more primitives than this are refitted by a block each, the rest
// by a warp each.
constexpr int kRefitBig = 1024;

struct BatchArgs;

// Bidirectional estimator (light-tracer connections + camera samples with next-event
// estimation, balance heuristic): counts N (light paths of the estimator) and M (camera
// samples), the camera samples' optional mask and decision hashes.
struct BidirArgs {
  float N, M;
  int64_t n_cam;
  const uint8_t* cam_mask;
  uint32_t* cam_hash;
};

// Kernel launchers.  lt_kernels.cu is compiled once per BVH width into namespaces w2, w4
// and w8; the functions of the same names in lt itself pick the variant by the scene's
// width (DevScene::width).
#define LT_KERNEL_LAUNCHERS                                                                                        \
  cudaError_t launch_refit(const RefitArgs& a, cudaStream_t st);                                                  \
  cudaError_t launch_primal(const DevScene& S, const KParams& kp, int est, float* image, void* aux,               \
                            const LaunchCfg& L, cudaStream_t st);                                                 \
  /* the plain primal's path order (KParams::order), `area`: the sort's work area of the state */                  \
  cudaError_t launch_path_order(const DevScene& S, const KParams& kp, unsigned* area, cudaStream_t st);            \
  cudaError_t launch_lrb3(const DevScene& S, const KParams& kp, bool att, bool chains, const float* dI,           \
                          const GradPtrs& g, void* state, bool mask_ready, const LaunchCfg& L, cudaStream_t st);  \
  cudaError_t launch_reslrb(const DevScene& S, const KParams& kp, bool att, bool chains, const float* dI,         \
                            const void* rec, const GradPtrs& g, const LaunchCfg& L, cudaStream_t st);             \
  cudaError_t launch_naive(const DevScene& S, const KParams& kp, bool att, bool chains, const float* dI,           \
                           const void* ws, const GradPtrs& g, const LaunchCfg& L, cudaStream_t st);               \
  cudaError_t launch_lrb2_reduce(const DevScene& S, const KParams& kp, const float* dI, void* buf,                \
                                 const GradPtrs& g, const LaunchCfg& L, cudaStream_t st);                         \
  cudaError_t launch_lrb2(const DevScene& S, const KParams& kp, bool att, bool chains, const float* dI,           \
                          void* buf, const GradPtrs& g, const LaunchCfg& L, cudaStream_t st);                     \
  cudaError_t launch_collect(const DevScene& S, const KParams& kp, const float* dI, float tfloor, float* feats,   \
                             float* targets, int64_t cap, unsigned long long* count, const LaunchCfg& L,          \
                             cudaStream_t st);                                                                    \
  /* sum of the copies of the albedo gradient (KParams::rep), and of KParams::le_sum if there is one */            \
  cudaError_t launch_rep_sum(const DevScene& S, const KParams& kp, int n_mats, const GradPtrs& g, cudaStream_t st); \
  cudaError_t launch_film_l2(const float* I, const float* T, int64_t n, float* dI, float* loss, int sms,          \
                             cudaStream_t st);                                                                    \
  cudaError_t launch_bidir(const DevScene& S, const KParams& kp, const BidirArgs& ba, bool backward, float* image, \
                           const float* dI, const GradPtrs& g, const LaunchCfg& L, cudaStream_t st);             \
  cudaError_t launch_lrb3_literal(const DevScene& S, const KParams& kp, const float* dI, const GradPtrs& g,       \
                                  const LaunchCfg& L, cudaStream_t st);

namespace w2 { LT_KERNEL_LAUNCHERS }
namespace w4 { LT_KERNEL_LAUNCHERS }
namespace w8 { LT_KERNEL_LAUNCHERS }
LT_KERNEL_LAUNCHERS

// `state` of launch_lrb3 (or null: fused kernel): per-path state of the two-kernel form.
//  - a record of 32 B per path (at 0), eight words.  The plain primal keeps there, for a path
//    with a valid connection, the primitives of its first vertices (HitBits, packed from bit 0
//    upwards), so that the passes intersect the known primitive instead of searching the scene.
//    A path with several valid connections has words 0-4 for them, and words 5-7 are pass 2's,
//    for delta_total; a path with one has words 0-2, and words 3-7 hold the film position and the
//    contribution (u_x, u_y, L.rgb) of that connection, from which pass 3 forms delta_total
//    itself.  Pass 2 overwrites nothing that the primal recorded (where it traces the
//    connections itself it writes the same one), so any number of backward calls, with other
//    image adjoints, may follow one primal.  One aligned sector per path, because the passes
//    visit the paths in the order of the list and gather it.
//  - validity bits 0-31 (at lrb3_state_mlo) and 32-63 (at lrb3_state_mhi), uint32 each; with a
//    depth of at most 32 the second word continues the recorded primitives instead (after word 2
//    or word 4 of the record);
//  - the list of the paths that have a valid connection (uint32 indices relative to the call, at
//    lrb3_state_list), written by the plain primal so that passes 2 and 3 visit only those, and
//    256 B of counters at lrb3_state_count: its length, the passes' counters of entries taken
//    (two), the number of listed paths with several connections, the number of paths in the order
//    (uint64 each), then KParams::le_sum; while the order is built, the list's place holds the
//    paths' sort keys;
//  - the order in which the plain primal takes the paths (uint32[n_paths] at lrb3_state_order;
//    the backward reuses the array for the listed paths with several connections) and the
//    counting sort's work area that builds it (kSortBins x kSortBlocks counts, then kSortBins
//    bin starts).
// In all 48 B per path, flat in depth.
constexpr int kSortBins = 4096;   // 64 x 64 cells of the first direction
constexpr int kSortBlocks = 256;  // blocks of the sort, each over a contiguous range of paths
__host__ __device__ inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
__host__ __device__ inline size_t lrb3_state_mlo(int64_t n) { return align256((size_t)n * 32); }
__host__ __device__ inline size_t lrb3_state_mhi(int64_t n) { return lrb3_state_mlo(n) + align256((size_t)n * 4); }
__host__ __device__ inline size_t lrb3_state_core(int64_t n) { return lrb3_state_mhi(n) + align256((size_t)n * 4); }
__host__ __device__ inline size_t lrb3_state_list(int64_t n) { return lrb3_state_core(n); }
__host__ __device__ inline size_t lrb3_state_count(int64_t n) { return lrb3_state_list(n) + align256((size_t)n * 4); }
__host__ __device__ inline size_t lrb3_state_order(int64_t n) { return lrb3_state_count(n) + 256; }
__host__ __device__ inline size_t lrb3_state_sort(int64_t n) { return lrb3_state_order(n) + align256((size_t)n * 4); }
__host__ __device__ inline size_t lrb3_state_bytes(int64_t n) {
  return lrb3_state_sort(n) + align256(sizeof(unsigned) * (size_t)kSortBins * (kSortBlocks + 1));
}
// The per-path arrays of a state (or of the buffered two-pass buffer) of n paths: words 0-3 and
// 4-7 of the record of path p are at a[step * p] and b[step * p].
struct PathState {
  float4 *a, *b;
  uint32_t *mlo, *mhi;
  int step;
};
__host__ __device__ inline PathState path_state(void* base, int64_t n) {
  char* c = (char*)base;
  return PathState{(float4*)c, (float4*)c + 1, (uint32_t*)(c + lrb3_state_mlo(n)), (uint32_t*)(c + lrb3_state_mhi(n)), 2};
}
// The path list is used for calls of at most this many paths (uint32 indices).
constexpr int64_t kListMaxPaths = 0xffffffffll;

// Buffer of the buffered two-pass estimator (lrb_2pass): per path words 4-7 of an LRB-3 record
// (16 B), validity bits 32-63 and its traced vertex count (int), then per vertex [depth][path]
// the splat record (u_x, u_y, L.r, L.g) (float4; u_x < 0 = no valid connection) and L.b
// (float), then per path words 0-3 of the record and validity bits 0-31, then the backward's
// copies of the albedo gradient (at most 4 MB; the splat records stay as the primal wrote them, so
// that any number of backward calls may follow it).
struct Lrb2Layout {
  size_t mhi, counts, rec4, recz, rec0, mlo, rep, total;
};
__host__ __device__ inline Lrb2Layout lrb2_layout(int64_t n, int d) {
  Lrb2Layout L;
  L.mhi = align256((size_t)n * 16);
  L.counts = L.mhi + align256((size_t)n * 4);
  L.rec4 = L.counts + align256((size_t)n * 4);
  L.recz = L.rec4 + align256((size_t)n * (size_t)d * 16);
  L.rec0 = L.recz + align256((size_t)n * (size_t)d * 4);
  L.mlo = L.rec0 + align256((size_t)n * 16);
  L.rep = L.mlo + align256((size_t)n * 4);
  const size_t most = (size_t)4 << 20, rep = (size_t)n * (size_t)d * 16;
  L.total = L.rep + align256(rep < most ? rep : most);
  return L;
}
__host__ __device__ inline PathState lrb2_path_state(void* buf, int64_t n, int d) {
  const Lrb2Layout L = lrb2_layout(n, d);
  char* c = (char*)buf;
  return PathState{(float4*)(c + L.rec0), (float4*)c, (uint32_t*)(c + L.mlo), (uint32_t*)(c + L.mhi), 1};
}
size_t mlp_grad_smem_bytes();
cudaError_t launch_mlp_grad(const float* P, const float* X, const float* T, int64_t n, float inv_batch, float* g,
                            float* loss, int sms, cudaStream_t st);
cudaError_t launch_mlp_adam(float* P, float* M, float* V, const float* g, int step, float lr, cudaStream_t st);
cudaError_t launch_mlp_moments(const float* X, const float* T, int64_t n, float* P, cudaStream_t st);
cudaError_t launch_mlp_forward(const float* P, const float* X, int64_t n, float* out, int sms, cudaStream_t st);

}  // namespace lt
