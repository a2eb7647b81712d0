// Host-side model object behind the opaque js_model handle.
#pragma once
#include <cuda.h>

#include <vector>

#include "js_common.cuh"

// Tensor-core view of a masked MLP: per layer the output-tile width, the tile
// metadata (last live K block, smallest / largest degree) and the TMA descriptors.
struct TcLayer {
    const int *kb_end;
    const int *dmin;
    const int *dmax;
    int bn;
    int nt;
    int stage_bytes, n_stages;   // this layer's cut of the operand ring
    int npad;                    // units padded to whole tiles: rows per K block of the tile-major weight copy
    // split-K: the K blocks of tile nt are cut into chunks of `ch` blocks, each chunk a work unit
    // of its own; the last chunk owns the tile and adds the others' fp32 partial sums in order
    int ch;
    int slots_per_mt;            // partial-sum slots per row tile = sum over nt of (chunks - 1)
    const int *slot_base;        // [nt] first slot of tile nt inside a row tile
    int n_sched;                 // schedules: one per number of live row tiles (1..n_sched), or a single one
    const int *sched_off;        // [n_sched][grid + 1] work units of CTA c: sched[sched_off[c] .. sched_off[c+1])
    const int *sched;            // units packed as (row tile << 24) | (n tile << 8) | chunk
};
struct TcDev {
    const CUtensorMap *tmA;      // [L+1] activations a[l], box 64 x 128
    const CUtensorMap *tmW;      // [L+1] masked weights W[l], box 64 x bn
    TcLayer lay[JS_MAXL + 1];
    int stage_bytes, n_stages, smem_bytes;
    int ring_bytes, aux_bytes;   // shared memory: operand ring, then the epilogues' auxiliary buffer,
    int meta_bytes, ucap;        // tile metadata, decoded units (the first ucap of every layer)
    int cat_rows;                // 256-way outputs: the first cat_rows rows of a tile get their noise through shared memory
    int bin_bulk;                // binary output rows are 16-byte granular: moved by bulk copies
    int grid;                    // CTAs the schedules were built for (the launch uses exactly this)
    float *partials;             // [slot][columns/4][128 rows] float4: fp32 partial sums of non-owning chunks
    unsigned *pflags;            // [slot][4 row quadrants][2 column halves]: phase stamp once the partial is stored
    int n_pflags;
    bool streams;                // output weights that do not stay in L2 from pass to pass
};

// What the cached sweeps (made_sweep.cu) need beside the tensor-core view.
struct SweepDev {
    const CUtensorMap *tmAold;          // [3][L+1] activations a[l] of the previous iterate, boxes 64 x 32, 64, 128
    const CUtensorMap *tmF;             // [3][L+1] the jobs' buffers F[l], 3-D {column, row, slot}, boxes 64 x 32, 64, 128 x 1
    int rj, rj_idx;                     // sample rows per job (32 << rj_idx)
    const CUtensorMap *tmW16;           // [3][L+1] masked weights W[l]: boxes of 64 x 16, 64 x 32 and 64 x 64 (columns x rows)
    float *S;                           // [slot][L+1][nbs][128 rows] fp32: base sums of a job's next groups
    int nbs;
    __nv_bfloat16 *F[JS_MAXL + 1];      // [slot][128 rows][WF[l]]: a job's fresh activations of a[l]
    int WF[JS_MAXL + 1];
    const int *cnt[JS_MAXL + 1];        // cnt[l][d], d = 0..T: units of a[l] with degree <= d (l >= 1)
    int G;                              // positions per group
    int n_stages, ring_bytes, smem_bytes, slots;
};

// Small fp32 masked MLPs (made_small.cu): how a cluster of CS CTAs shares the units, and the packed weights.
#define SMALL_KENDS 16
struct SmallDev {
    int CS, cs_log2, sms;
    int nc[JS_MAXL + 1], ncs[JS_MAXL + 1];          // own outputs per CTA and layer, row stride of the packed weights
    int w_off[JS_MAXL + 1], b_off[JS_MAXL + 1], d_off[JS_MAXL + 1];     // float offsets inside a CTA's pack
    int kend[JS_MAXL + 1][SMALL_KENDS];             // last live input of every block of 32 own outputs
    int pack_floats;
    const float *pack;                              // [CS][pack_floats]
};

// Binary bf16 models on the cluster kernel (made_cluster.cu): tiles of 64 units per layer.
#define CL_MAXL 3             // hidden layers
#define CL_TILES 48           // tiles (and K blocks) per layer
struct ClTiles {
    unsigned char kbe[CL_MAXL + 1][CL_TILES];       // K blocks a tile reads
    short dmin[CL_MAXL + 1][CL_TILES], dmax[CL_MAXL + 1][CL_TILES];
};
struct ClusterDev {
    int CS, cs_log2, max_clusters;
    int nt[CL_MAXL + 1], nkb[CL_MAXL + 1], npad[CL_MAXL + 1];
    int own_out;                 // most output tiles of one CTA
    int kblocks;                 // K blocks of weights a CTA reads per pass
    int early_ok;                // encodings may be sent as soon as they are sampled
    int n_stages;
    unsigned char need[CL_MAXL + 1][8], off[CL_MAXL + 1][8];     // per layer and CTA: K blocks of a[l] that it reads, where it keeps them
    int blocks;                  // most K blocks of activations in a CTA
    ClTiles tiles;
    const CUtensorMap *tmW;      // [L+1][2] tile-major weights: one K block of 64 units, two of them
};

// Device view of a masked-convolution stack (tensor-core kernel only).
struct ConvDev {
    int height, width, in_ch, ch, n_conv, C, T;
    int R;                              // image rows per 128-pixel tile
    int nyt;                            // row tiles per image
    int cin_pad[JS_MAXL];               // input channels of conv layer l, padded to a multiple of 64
    void *act[JS_MAXL + 1];             // NHWC bf16; act[0] = encoded image padded to 64 channels
    void *act_old[JS_MAXL + 1];         // the same for the previous outer iterate (Jacobi-GS)
    const float *bias[JS_MAXL + 1];     // conv biases, head bias at [n_conv]
    const float *lut;
    int *stamp;                         // [batch][nyt][8]: number of the last layer that wrote each eighth of a tile
    const CUtensorMap *tmAct;           // [n_conv+1] 4-D maps {channel, x, y, image}, box 64 x width x R x 1
    const CUtensorMap *tmActOld;        // the same over act_old
    const CUtensorMap *tmAct2, *tmActOld2;      // the same with boxes of R + 1 rows
    int share, stage_a;                 // conv layers load R + 1 rows at once; bytes of a pixel stage
    const CUtensorMap *tmW;             // [n_conv+1] 2-D maps of the packed weights
};

#define JS_MAX_CLUSTERS 4096          // most clusters a call of the cluster kernels may have

// What a launch of a cluster kernel consists of, for the statistics.
struct ClusterWork {
    int clusters;
    int tiles;                              // output tiles of a pass, all layers (cluster kernel of bf16 models)
    long long block_flops, block_bytes;     // of a K block: its MMAs, its weights
};

struct js_model {
    std::vector<int> host_kend[JS_MAXL + 1];       // t_kend of the device view
    int kind = 0;                 // 0 masked MLP, 1 masked-conv stack
    int max_batch = 0;
    int rows = 0;                 // max_batch rounded up to a multiple of 128
    MadeDev made{};
    int conv_T = 0, conv_C = 0;
    std::vector<void *> allocs;   // every device allocation, freed by js_model_destroy
    std::vector<std::vector<int>> host_deg;
    JsCtl *ctl = nullptr;
    JsCtl *h_result = nullptr;    // pinned host memory, mapped: the kernels report here
    JsCtl *d_result = nullptr;    // the same memory as the device sees it
    unsigned long long *h_words = nullptr, *d_words = nullptr;      // JS_MAX_CLUSTERS reports of two words, mapped like h_result
    bool ctl_clean = false;       // the last call left the control block zeroed
    // host-buffer entry point: device staging, copy stream, "noise has arrived" word
    float *st_noise = nullptr;
    uint8_t *st_x = nullptr, *st_init = nullptr;
    int32_t *st_iters = nullptr;
    unsigned *d_nflag = nullptr, *h_nflag = nullptr;
    unsigned n_uploads = 0;
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t ev_main = nullptr, ev_copy = nullptr;
    int *smp_changed = nullptr, *smp_state = nullptr, *perm = nullptr;
    uint8_t *x_old = nullptr, *x_tmp = nullptr;
    unsigned long long *trace = nullptr;
    int opt_frontier_skip = 1, opt_seq_skip = 2, opt_spin_limit = 1 << 22, opt_path = 0, opt_compact = 1, opt_trace = 0;
    int max_grid_generic[3] = {0, 0, 0};   // of the products' instance, of Jacobi-GS's, of the products with split inputs
    TcDev tc{};
    int tc_ok = 0, tc_max_grid = 0;
    const void *tc_weights[JS_MAXL + 1] = {};       // tile-major weights of the tensor-core kernels
    ClusterDev cluster{};
    int cluster_ok = 0;
    SmallDev small{};
    int small_ok = 0;
    ConvDev conv{};
    int conv_max_grid = 0;
    SweepDev sweep{};
    int sweep_state = 0;          // 0 not prepared yet, 1 ready, -1 the model does not qualify
    int *sw_flags = nullptr;      // [2][rows]: per-sample change flags and done flags of the sweeps
    int *h_any = nullptr, *d_any = nullptr;      // mapped host word: did anything change in this outer iteration
    js_stats stats{};
};

int js_tc_prepare(js_model *m);
int js_launch_made_tc(const js_model *m, const RunArgs &r, cudaStream_t stream);
int js_small_prepare(js_model *m);
bool js_small_serves(const js_model *m, const RunArgs &r);
int js_launch_made_small(const js_model *m, const RunArgs &r, cudaStream_t stream, ClusterWork *work);
bool js_tensor_maps();        // can the driver encode them?
bool js_encode_map(CUtensorMap *out, CUtensorMapDataType type, const void *base, int rank, const cuuint64_t *dims,
                   const cuuint64_t *strides, const cuuint32_t *box);
bool js_encode_map_2d(CUtensorMap *out, CUtensorMapDataType type, const void *base, int rows, int cols, int box_cols, int box_rows,
                      int row_stride = 0);
int js_generic_prepare(js_model *m);
int js_cluster_prepare(js_model *m);
bool js_cluster_serves(const js_model *m, const RunArgs &r);
int js_launch_made_cluster(const js_model *m, const RunArgs &r, cudaStream_t stream, ClusterWork *work);
int js_conv_build(js_model *m, const js_conv_desc *d);
int js_launch_conv_tc(const js_model *m, const RunArgs &r, cudaStream_t stream);
int js_sweep_prepare(js_model *m);
int js_launch_made_sweep(const js_model *m, const RunArgs &r, cudaStream_t stream);
int js_launch_jgs_book(const js_model *m, int batch, int k, int at_cap, int32_t *out_iters, cudaStream_t stream);
