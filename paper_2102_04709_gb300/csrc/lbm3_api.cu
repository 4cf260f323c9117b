// lbm3_api.cu -- host side of the C ABI declared in include/lbm3.h: argument checks, node
// classification (Section II.B), eighth-order solid normals (Eq.19-20), the compact wall list,
// device buffers and the per-step launch sequence.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include <sys/mman.h>
#include <unistd.h>

#include <cudaTypedefs.h>

#include "../../include/lbm3.h"
#include "lbm3_common.cuh"

using namespace lbm3k;

struct lbm3 {
    Params P{};
    int precision = 0;
    cudaStream_t stream = nullptr;
    // device buffers: two population buffers (FP32 planes, or FP32 densities + 16-bit offset
    // planes), the node classes, wall values, velocity, scratch
    Pop pop[2] = {{nullptr, nullptr, nullptr}, {nullptr, nullptr, nullptr}};
    uint8_t* type = nullptr;
    // [3][N] wall values (a step writes C_SB nodes only); cw[pp] are the current ones
    double* cw[2] = {nullptr, nullptr};
    float* u = nullptr;
    double* scratch = nullptr;     // 3N: rho, then u, as lbm3_fields returns them
    double* partials = nullptr;    // diagnostics block partials
    double* dout = nullptr;        // 8 doubles
    int* err_flag = nullptr;       // error bits set by kernels (Params::err)
    // bulk-tensor-copy path of the pure tiles (nx a multiple of 4): tensor maps of each
    // population buffer, FP32 storage: the two parts of the source box and the destination tile;
    // 16-bit storage: the density box (tm_in_a) and the offset-plane box (tm_in_b)
    bool tma = false;
    // blocks of the persistent pure-tile kernel, and the index in use: [1] where so many pure tiles are
    // its own that it needs the SMs that [0] leaves to launch_step_one (the same where that is not
    // launched); see count_tiles
    int pure_blocks[2] = {0, 0};
    int many = 0;
    unsigned *count_dev = nullptr, *count_host = nullptr;  // its tiles when last counted (host: pinned)
    int count_limit = 0, count_age = 0;                    // [1] from this many on; steps since the count
    CUtensorMap tm_in_a[2], tm_in_b[2], tm_out[2];
    // FP32 pure tiles through the ring kernel (one producer warp, two consumer groups, one block
    // per SM): tensor maps of each buffer with the whole pull box
    bool ring = false;
    CUtensorMap tm_box[2];
    int* widx = nullptr;
    double* wnrm = nullptr;
    float* wang = nullptr;
    // set by the adjoint for one step: the step reads io_in (through the tensor map io_box on the
    // ring path) and writes io_out instead of the two population buffers, whose turn is kept
    const Pop* io_in = nullptr;
    const Pop* io_out = nullptr;
    double* io_cw_out = nullptr;  // and its wall values go there
    const CUtensorMap* io_box = nullptr;
    // the timing events of enqueue_step are recorded into a graph being captured (as nodes that
    // record them when the graph runs)
    bool ev_external = false;
    int nw = 0;
    long long n_fluid = 0;
    // tiles of the step kernels: gen, those near solids or the domain edge (launch_tile, on a
    // higher-priority side stream), then the pure ones (no solid within 3 nodes, away from the edge;
    // main stream)
    TileSet gen{};
    int n_pure = 0, n_gen = 0;
    const int* tiles_pure = nullptr;
    void* tile_mem[5] = {};  // the arrays of the set, and the pure tiles' list
    int n_went = 0;          // entries of the wetting (gen.went), four lanes of its cache each
    long long pure_fluid = 0;
    // a word per tile, what its rows hold (one byte per row, written by one warp, so no byte needs an
    // atomic or a clearing): pres[pp] describes the current state, and every launch of a step writes the
    // next one's for the tiles that it advances (launch_step_tma, which does not look what they hold, as
    // 0x07: all fluids), so that a run may go from one set of launches to another between any two steps.
    // All words say 0x07 after the state is replaced from outside, those of tiles without a fluid node
    // for ever.  While pp == cur, pres[b] describes buffer pop[b]: the planes of a fluid that a tile's
    // word does not name hold zeros there, which launch_step_one relies on to leave them unwritten.  pp
    // turns with cur (and alone in the adjoint's slot-to-slot steps, which therefore write every plane).
    uint64_t* pres[2] = {nullptr, nullptr};
    size_t pres_bytes = 0;
    int pp = 0;
    cudaStream_t side = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    // chain: a small grid, every tile in one launch per step (kChainTiles); the records of the pure
    // tiles then follow those of gen
    bool chain = false;
    // one: the pure tiles with one fluid around are launch_step_one's (kOneTiles); those with
    // several run beside them on a third side stream
    bool one = false;
    cudaStream_t side3 = nullptr;
    cudaEvent_t ev_join3 = nullptr;
    // CUDA graphs of kGraphSteps consecutive steps (an even count: a graph starts and ends on the
    // same population buffer), one per starting buffer (and launch size), captured on the internal stream gcap
    // when lbm3_step first needs them and replayed on the caller's stream; dropped when a
    // captured launch argument changes (lbm3_set_inflow).  graph_off: a capture failed, so steps
    // are launched one by one (the same kernels, the same results).
    cudaStream_t gcap = nullptr;
    cudaGraphExec_t gexec[2][2] = {};  // by `many` and starting buffer
    bool graph_off = false;
    size_t bytes = 0;
    int cur = 0;
    bool ready = false;
    std::vector<int> wall_host;
    std::string err;
    // device memory of lbm3_adjoint_centroid, kept for later calls that need no more of it: the
    // checkpoints (nck states), the segment's states (nsg), the final state and the work arrays;
    // released by lbm3_adjoint_release or
    // lbm3_destroy
    struct AdjStore {
        float *ck_f = nullptr, *sg_f = nullptr, *fin_f = nullptr;
        double *ck_c = nullptr, *sg_c = nullptr, *fin_c = nullptr;
        int nck = 0, nsg = 0;
        AdjointWork* W = nullptr;
        std::vector<CUtensorMap> box;  // ring path: the tensor map of every segment slot
        // the sweep as a graph, for nsteps / K from state buffer g_cur
        cudaGraphExec_t gexec = nullptr;
        int g_nsteps = 0, g_K = 0, g_cur = 0;
    } adj;
};

namespace {

std::string g_create_error;

int fail(lbm3* h, int code, const std::string& msg)
{
    if (h) h->err = msg; else g_create_error = msg;
    return code;
}

#define CUDA_TRY(h, call)                                                              \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess)                                                         \
            return fail(h, e_ == cudaErrorMemoryAllocation ? LBM3_ERR_OOM : LBM3_ERR_CUDA, \
                        std::string(#call) + ": " + cudaGetErrorString(e_));           \
    } while (0)

// Solid indicator s(x) of Eq.(19) at an unwrapped position: periodic sides wrap, wall sides
// are solid beyond the domain, open sides are fluid beyond the domain.
struct Indicator {
    int nx, ny, per_y, bc_x;
    const uint8_t* m;
    int operator()(int X, int Y) const
    {
        if (Y < 0 || Y >= ny) {
            if (!per_y) return 1;
            Y = ((Y % ny) + ny) % ny;
        }
        if (X < 0 || X >= nx) {
            if (bc_x == kWalls) return 1;
            if (bc_x == kZouHe) return 0;
            X = ((X % nx) + nx) % nx;
        }
        return m[(size_t)Y * nx + X] ? 1 : 0;
    }
    bool outside_solid(int X, int Y) const
    {
        if ((Y < 0 || Y >= ny) && !per_y) return true;
        if ((X < 0 || X >= nx) && bc_x == kWalls) return true;
        return false;
    }
};

// g(X) of Eq.(15)
double seg_g(double X)
{
    if (X < -1.0) return 1.0;
    if (X > 1.0) return -1.0;
    const double s = std::sqrt(std::max(0.0, 1.0 - X * X));  // sin(arccos X)
    return X < 0.0 ? 1.0 - s : s - 1.0;
}

size_t tally(lbm3* h, size_t b)
{
    h->bytes += b;
    return b;
}

void adj_release(lbm3* h)
{
    lbm3::AdjStore& a = h->adj;
    void* ptrs[] = {a.ck_f, a.sg_f, a.fin_f, a.ck_c, a.sg_c, a.fin_c};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    if (a.gexec) cudaGraphExecDestroy(a.gexec);
    adjoint_free(a.W);
    a = lbm3::AdjStore{};
}

void release(lbm3* h)
{
    adj_release(h);
    void* ptrs[] = {h->pop[0].f, h->pop[1].f, h->pop[0].rho, h->pop[1].rho, h->pop[0].off,
                    h->pop[1].off, h->type, h->cw[0], h->cw[1], h->u, h->scratch, h->partials, h->dout,
                    h->widx, h->wnrm, h->wang, h->err_flag, h->gen.cache, h->pres[0], h->pres[1], h->count_dev,
                    h->tile_mem[0], h->tile_mem[1], h->tile_mem[2], h->tile_mem[3], h->tile_mem[4]};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    h->pop[0] = h->pop[1] = Pop{nullptr, nullptr, nullptr};
    if (h->count_host) cudaFreeHost(h->count_host);
    for (int c = 0; c < 4; c++)
        if (h->gexec[c / 2][c % 2]) cudaGraphExecDestroy(h->gexec[c / 2][c % 2]);
    if (h->gcap) cudaStreamDestroy(h->gcap);
    if (h->ev_fork) cudaEventDestroy(h->ev_fork);
    if (h->ev_join) cudaEventDestroy(h->ev_join);
    if (h->ev_join3) cudaEventDestroy(h->ev_join3);
    if (h->side3) cudaStreamDestroy(h->side3);
    if (h->side) cudaStreamDestroy(h->side);
}

// From this many pure tiles on, the tiles with one fluid around are launch_step_one's, and the pure ones
// with several run beside them on a stream of their own.  On smaller grids the fluids soon reach every
// tile, the step waits for the tiles near solids, and two more launches cost more than they hide.  us a step
// with them and without, after 300, 1500 and 6000 steps: the 512 x 512 cylinder (803 pure tiles) 22.9 22.9
// 23.0 / 18.5 19.2 19.3, a 544 x 544 one (920) 23.0 25.4 25.5 / 20.5 21.9 22.0, the 800 x 375 pillars (865)
// 20.1 21.6 27.0 / 22.7 24.0 26.1 (one launch of all tiles 20.2 21.4 23.7), the 1030 x 517 ones (1571) 26.5
// 30.4 38.1 / 32.7 34.7 36.2, a 1024 x 1024 cylinder (3715) 36.8 40.0 58 / 55.7 57.7 60.7.
// LBM3_ONE_TILES=<n> in the environment at lbm3_create sets another line (same results).
constexpr int kOneTiles = 1200;

// Tiles up to which a step is one launch of all of them (k_tile, two blocks per SM: four rounds of
// blocks), one launch behind the other with no fork to the side streams and no join, and the start of a
// step (its record, the geometry words) under the end of the one before (programmatic dependent launch).
// Beyond, k_tile's time for a pure tile counts: us a step with the launches beside one another and with
// one, after 300, 1500 and 6000 steps: 128 x 64 16.9 17.0 16.9 / 15.5 15.2 15.2, 450 x 31 19.0 18.8 19.7 /
// 17.6 17.3 17.8, 2048 x 128 (1024 tiles) 17.6 17.7 19.7 / 17.5 17.7 17.8, the 512 x 512 cylinder (1024) 18.5
// 19.2 19.3 / 18.7 19.9 20.0, a 544 x 544 one (1156) 20.5 21.9 22.0 / 19.7 21.8 22.1, the 800 x 375 pillars
// (1175) 22.7 24.0 26.1 / 20.2 21.4 23.7, the 1030 x 517 ones (2145) 32.7 34.7 36.2 / 35.0 39.6 46.7.
// LBM3_CHAIN_TILES=<n> in the environment at lbm3_create sets another line (same results).
constexpr int kChainTiles = 1200;

// Tensor maps of one [27][ny][nx] FP32 population buffer: as the two parts of the pull-source box
// of a pure tile, (kTX + 8) x (kTY + 6) x kTmaPlanesA and x (27 - kTmaPlanesA) planes, and as its
// destination tile kTX x kTY x 27.  false if the driver has no encoder or refuses the layout (the
// plain kernel is used then).
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn) {
            cudaGetLastError();
            return nullptr;
        }
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    return encode;
}

// Tensor map of one [27][ny][nx] FP32 population buffer with the whole pull box of a pure tile,
// (kTX + 8) x (kTY + 6) x 27, for the ring kernel.
bool make_box_map(const Params& P, float* f, CUtensorMap* box)
{
    const PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
    if (!encode) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)P.nx, (cuuint64_t)P.ny, 27};
    const cuuint64_t strides[2] = {(cuuint64_t)P.nx * sizeof(float), (cuuint64_t)P.N * sizeof(float)};
    const cuuint32_t bx[3] = {kTX + 8, kTY + 6, 27};
    const cuuint32_t unit[3] = {1, 1, 1};
    return encode(box, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, f, dims, strides, bx, unit, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_tensor_maps(const Params& P, float* f, CUtensorMap* in_a, CUtensorMap* in_b, CUtensorMap* out)
{
    const PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
    if (!encode) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)P.nx, (cuuint64_t)P.ny, 27};
    const cuuint64_t strides[2] = {(cuuint64_t)P.nx * sizeof(float), (cuuint64_t)P.N * sizeof(float)};
    const cuuint32_t box_a[3] = {kTX + 8, kTY + 6, kTmaPlanesA};
    const cuuint32_t box_b[3] = {kTX + 8, kTY + 6, 27 - kTmaPlanesA};
    const cuuint32_t box_out[3] = {kTX, kTY, 27};
    const cuuint32_t unit[3] = {1, 1, 1};
    auto enc = [&](CUtensorMap* m, const cuuint32_t* box) {
        return encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, f, dims, strides, box, unit,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    return enc(in_a, box_a) && enc(in_b, box_b) && enc(out, box_out);
}

// Tensor maps of one 16-bit-storage population buffer: the densities rho[3][ny][nx] (FP32, box
// (kTX + 8) x (kTY + 6) x 3) and the offset planes off[24][ny][nx] (16-bit words, box
// (kTX + 16) x (kTY + 6) x 24; its row pitch 2 nx bytes must be a multiple of 16).
bool make_tensor_maps16(const Params& P, const Pop& p, CUtensorMap* trho, CUtensorMap* toff)
{
    const PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
    if (!encode) return false;
    const cuuint64_t rdims[3] = {(cuuint64_t)P.nx, (cuuint64_t)P.ny, 3};
    const cuuint64_t rstrides[2] = {(cuuint64_t)P.nx * sizeof(float), (cuuint64_t)P.N * sizeof(float)};
    const cuuint32_t rbox[3] = {kTX + 8, kTY + 6, 3}, unit[3] = {1, 1, 1};
    const cuuint64_t odims[3] = {(cuuint64_t)P.nx, (cuuint64_t)P.ny, 24};
    const cuuint64_t ostrides[2] = {(cuuint64_t)P.nx * 2, (cuuint64_t)P.N * 2};
    const cuuint32_t obox[3] = {kTX + 16, kTY + 6, 24};
    return encode(trho, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, p.rho, rdims, rstrides, rbox, unit,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS &&
           encode(toff, CU_TENSOR_MAP_DATA_TYPE_UINT16, 3, p.off, odims, ostrides, obox, unit,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// a timing event of enqueue_step (a record node when captured into a graph)
void record_timing(lbm3* h, cudaEvent_t ev, cudaStream_t s)
{
    if (h->ev_external)
        cudaEventRecordWithFlags(ev, s, cudaEventRecordExternal);
    else
        cudaEventRecord(ev, s);
}

// polls of an mbarrier before a step kernel gives up on a tile's bulk copies (a completed copy
// takes a few microseconds; this is seconds of polling)
constexpr int kCopyWaitPolls = 1 << 22;

// whether a step is one launch of every tile.  A lowered copy-wait limit is for the bulk copies of the
// other launches.
bool chained(const lbm3* h) { return h->chain && h->P.wait_polls == kCopyWaitPolls; }

// One timestep: fork the side streams off the main stream, run the pure tiles on the main stream
// (those with several fluids around on a side stream of their own where launch_step_one takes the
// others) and the other tiles, with the wetting of their solid boundary nodes, on the
// higher-priority side stream; join.  With ev != NULL the launches of such a step are bracketed by events
// (main stream: ev[0], ev[1], the pure tiles; side stream: ev[2], ev[3], the others).
cudaError_t enqueue_step(lbm3* h, bool last, cudaEvent_t* ev)
{
    cudaError_t e;
    const bool io = h->io_in != nullptr;
    const Pop& fin = io ? *h->io_in : h->pop[h->cur];
    const Pop& fo = io ? *h->io_out : h->pop[1 - h->cur];
    double* cw_out = io ? h->io_cw_out : h->cw[1 - h->pp];
    float* u = last ? h->u : nullptr;
    const uint64_t* pin = h->pres[h->pp];
    uint64_t* pout = h->pres[1 - h->pp];
    if (chained(h)) {
        // a small grid: every tile in one launch, one step behind the other on the main stream
        TileSet all = h->gen;
        all.ntiles = h->n_gen + h->n_pure;
        e = launch_tile(h->precision, h->P, all, fin, fo, cw_out, u, pin, pout, io, false, true, h->stream);
        if (!io) h->cur = 1 - h->cur;
        h->pp = 1 - h->pp;
        return e;
    }
    if ((e = cudaEventRecord(h->ev_fork, h->stream)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(h->side, h->ev_fork, 0)) != cudaSuccess) return e;
    if (ev) record_timing(h, ev[2], h->side);
    // steps between the adjoint's slots write every plane and wall value: the tiles all of theirs
    const bool light = h->one && !io;
    e = launch_tile(h->precision, h->P, h->gen, fin, fo, cw_out, u, pin, pout, io, light, false, h->side);
    if (e != cudaSuccess) return e;
    // (behind the tiles that take long: in front of them, or of the pure tiles on either stream, it delays
    // what the step waits for, 5-10 % on the 2048 x 1024 pillars)
    if (light) launch_step_one(h->precision, h->P, h->gen, nullptr, 0, fin, fo, u, pin, pout, false, h->side);
    if (ev) record_timing(h, ev[3], h->side);
    if (ev) record_timing(h, ev[0], h->stream);
    // pure tiles: those with several fluids around through the kernel of the storage and layout,
    // those with one (launch_step_one) beside it; the two-blocks-per-SM kernel takes them all
    if (h->n_pure > 0 && h->tma && h->precision == LBM3_FP32 && !h->ring) {
        launch_step_tma(h->P, h->tiles_pure, h->n_pure, h->pure_blocks[h->many], fo, u, h->tm_in_a[h->cur],
                        h->tm_in_b[h->cur], h->tm_out[1 - h->cur], pout, h->stream);
    } else if (h->n_pure > 0) {
        const bool one = h->one;
        cudaStream_t ms = one ? h->side3 : h->stream;
        if (one && (e = cudaStreamWaitEvent(ms, h->ev_fork, 0)) != cudaSuccess) return e;
        if (h->ring)
            launch_step_ring(h->P, h->tiles_pure, h->n_pure, h->pure_blocks[h->many], fo, u,
                             io ? *h->io_box : h->tm_box[h->cur], pin, pout, !one, ms);
        else if (h->tma)
            launch_step_tma16(h->precision, h->P, h->tiles_pure, h->n_pure, h->pure_blocks[h->many], fo, u,
                              h->tm_in_a[h->cur], h->tm_in_b[h->cur], pin, pout, !one, ms);
        else
            launch_step_plain(h->precision, h->P, h->tiles_pure, h->n_pure, fin, fo, u, pin, pout, !one, ms);
        if (one) {
            TileSet none = h->gen;
            none.ntiles = 0;
            launch_step_one(h->precision, h->P, none, h->tiles_pure, h->n_pure, fin, fo, u, pin, pout, io, h->stream);
            if ((e = cudaEventRecord(h->ev_join3, ms)) != cudaSuccess) return e;
            if ((e = cudaStreamWaitEvent(h->stream, h->ev_join3, 0)) != cudaSuccess) return e;
        }
    }
    if (ev) record_timing(h, ev[1], h->stream);
    if ((e = cudaEventRecord(h->ev_join, h->side)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(h->stream, h->ev_join, 0)) != cudaSuccess) return e;
    if (!io) h->cur = 1 - h->cur;
    h->pp = 1 - h->pp;
    return cudaGetLastError();
}

constexpr int kGraphSteps = 8;
// Error bits that the kernels set (bit 0: a bulk tensor copy outlived its wait), read after the
// stream has been synchronised and cleared once read, so that each timeout is reported once.
int take_kernel_error(lbm3* h)
{
    int bits = 0;
    cudaError_t e = cudaMemcpyAsync(&bits, h->err_flag, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e == cudaSuccess && bits) e = cudaMemsetAsync(h->err_flag, 0, sizeof(int), h->stream);
    if (e != cudaSuccess) return fail(h, LBM3_ERR_CUDA, std::string("error bits: ") + cudaGetErrorString(e));
    if (bits & 1) return fail(h, LBM3_ERR_CUDA, "a bulk tensor copy of the step kernel did not complete in time");
    return LBM3_OK;
}

// First touch of the pages of an output array: while the device still works on the steps before, instead
// of page by page in the middle of the copy with the device waiting.  The values stay: a call that fails
// later has not written to the array.  (Values widened by the device and copied straight to the caller's
// arrays, on the 4096 x 2048 grid behind 256 steps: 6.4 ms; as floats through a vector, widened by the
// host: 27.  128 x 64 behind 8 steps: 58 and 157 us; through pinned memory 52 there, but five times longer
// from 512 x 512 on.)
void touch_pages(double* p, size_t n)
{
    if (n == 0) return;
    const uintptr_t page = (uintptr_t)sysconf(_SC_PAGESIZE);
    const uintptr_t from = (uintptr_t)p / page * page, to = (uintptr_t)(p + n);
#ifdef MADV_POPULATE_WRITE
    // (small arrays mostly have their pages: 128 x 64 pays 2 us for the system calls)
    if (n > (1u << 17) && madvise((void*)from, to - from, MADV_POPULATE_WRITE) == 0) return;
#endif
    // else one word of each page, written with what it holds
    for (size_t i = 0; i < n; i += 4096 / sizeof(double)) {
        volatile uint64_t* w = reinterpret_cast<volatile uint64_t*>(p + i);
        *w = *w;
    }
}

// the state was replaced from outside: every tile may hold every fluid
cudaError_t pres_reset(lbm3* h)
{
    h->pp = h->cur;
    cudaError_t e = cudaSuccess;
    for (int b = 0; b < 2 && e == cudaSuccess; b++) e = cudaMemsetAsync(h->pres[b], 0x07, h->pres_bytes, h->stream);
    return e;
}

void drop_graphs(lbm3* h)
{
    for (int c = 0; c < 4; c++) {
        cudaGraphExec_t& g = h->gexec[c / 2][c % 2];
        if (g) cudaGraphExecDestroy(g);
        g = nullptr;
    }
    if (h->adj.gexec) cudaGraphExecDestroy(h->adj.gexec);
    h->adj.gexec = nullptr;
}

// kGraphSteps steps from the current buffer, none of them the last of an lbm3_step call (no
// velocity output): replay of the captured graph, captured first if needed.  Capturing only
// records the launches (nothing runs), on the internal stream, so the caller's stream may be any
// stream, the legacy default one included.
cudaError_t graph_block(lbm3* h)
{
    const int c = h->cur, pc = h->pp;
    cudaGraphExec_t& x = h->gexec[h->many][c];
    if (!x && !h->graph_off) {
        cudaStream_t user = h->stream;
        h->stream = h->gcap;
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamBeginCapture(h->gcap, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            cudaError_t el = cudaSuccess;
            for (int s = 0; s < kGraphSteps && el == cudaSuccess; s++) el = enqueue_step(h, false, nullptr);
            e = cudaStreamEndCapture(h->gcap, &g);
            if (el != cudaSuccess) e = el;
        }
        h->stream = user;
        h->cur = c;
        h->pp = pc;
        if (e == cudaSuccess) e = cudaGraphInstantiate(&x, g, 0);
        if (g) cudaGraphDestroy(g);
        if (e != cudaSuccess) {
            x = nullptr;
            h->graph_off = true;
            cudaGetLastError();  // a failed capture leaves no sticky error; clear the last one
        }
    }
    if (!x) {
        for (int s = 0; s < kGraphSteps; s++) {
            const cudaError_t e = enqueue_step(h, false, nullptr);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    return cudaGraphLaunch(x, h->stream);  // ends on buffer c again
}

// Classes and flags of the nodes of a row but for its ends, with rows on either side: nine plain reads each
// (with the boundaries' rules for each of them this was most of a set-up).  Returns the fluid nodes.  (Out of
// line, where the compiler makes vectors of it: as a part of lbm3_create, which takes 29 ms on 4096 x 2048
// instead of 59, it took 24 ms of it or 37, with what else that function held.)
__attribute__((noinline)) long long classify_inside(const uint8_t* __restrict__ m, int nx, uint8_t* __restrict__ cls,
                                                    uint16_t* __restrict__ nflag)
{
    int n_fluid = 0;
    for (int x = 1; x < nx - 1; x++) {
        const int me = m[x] != 0;
        int flag = 0, others = 0;
        for (int a = 1; a < kQ; a++) {
            const int other = m[x + ey(a) * nx + ex(a)] != 0;
            others += other;
            flag |= other << opp(a);  // what comes along opp(a) would come from there
        }
        const bool touch = others != (me ? kQ - 1 : 0);
        nflag[x] = (uint16_t)(me ? kNodeSolid : flag);
        cls[x] = (uint8_t)(me ? (touch ? kSB : kSI) : (touch ? kFB : kFI));
        n_fluid += !me;
    }
    return n_fluid;
}

// The persistent pure-tile kernel's blocks.  SMs left free for the other kernels of a step while it holds its
// own: where it takes all pure tiles, the other tiles' share of the step's work, in units of a pure tile's SM
// time (such a tile 1.8, 0.038 per C_SB node).  Where k_step_one takes most of them, half of the SMs (beside
// the 16-bit kernel 2/5), and 1/5 once more than 3/10 (1/5) of the pure tiles hold or have several fluids
// around.  us a step with 76 (60), 50 and 30 left, at the share that does:
//   FP32 4096 x 2048  0.07 159 165 169, 0.23 188 196 202, 0.30 210 211 216, 0.39 248 236 241
//   FP32 2048 x 1024  0.13 60 62 64, 0.26 69 70 72, 0.32 77 75 78, 0.50 103 97 98, 0.72 124 116 114
//   FP16 4096 x 2048  0.07 162 162 165, 0.19 188 188 190, 0.23 203 197 198, 0.35 262 239 230
//   FP16 2048 x 1024  0.13 63 64 64, 0.20 68 70 68, 0.27 77 78 75, 0.45 112 113 106
// and all of them, after 100,000 steps of FP32 4096 x 2048, 486 430 404 (457 before there was a k_step_one).
// LBM3_SPARE_SMS=<n> in the environment at lbm3_create sets the count instead.
cudaError_t choose_blocks(lbm3* h, int sms)
{
    const bool f32 = h->precision == LBM3_FP32;
    const double wg = 1.8 * h->n_gen + 0.038 * h->nw;
    const int share = std::min(sms / 2, (int)std::lround(sms * wg / (wg + h->n_pure)));
    int spare[2] = {h->one ? (f32 ? sms / 2 : sms * 2 / 5) : share, h->one ? sms / 5 : share};
    if (const char* ov = std::getenv("LBM3_SPARE_SMS"))
        spare[0] = spare[1] = std::max(0, std::min(sms - 1, std::atoi(ov)));
    for (int b = 0; b < 2; b++)
        h->pure_blocks[b] = (f32 ? (h->ring ? 1 : kTmaBlocksPerSm) : kTma16BlocksPerSm) * (sms - spare[b]);
    if (spare[0] == spare[1]) return cudaSuccess;
    h->count_limit = (int)((long long)h->n_pure * (f32 ? 3 : 2) / 10);
    cudaError_t e = cudaMalloc((void**)&h->count_dev, sizeof(unsigned));
    if (e == cudaSuccess) tally(h, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMallocHost((void**)&h->count_host, sizeof(unsigned));
    if (e == cudaSuccess) *h->count_host = 0;
    return e;
}

// How many blocks the persistent kernel gets from here on.  The tiles that are its own grow in number for
// tens of thousands of steps, as the fluids' traces spread, and it needs more SMs then (pure_blocks); the
// blocks of a launch that find no tile cost nearly what the others cost.  So every kCountSteps steps or
// more its tiles are counted on the device, and the host takes the count that has arrived when it comes by:
// it never waits, an old one makes the steps no less right, and the two launches give the same bits.
constexpr int kCountSteps = 256;
cudaError_t count_tiles(lbm3* h, int steps)
{
    if (!h->count_host || chained(h)) return cudaSuccess;
    const unsigned n = *const_cast<volatile unsigned*>(h->count_host);
    h->many = n > (unsigned)h->count_limit;
    h->count_age += steps;
    if (h->count_age < kCountSteps) return cudaSuccess;
    h->count_age = 0;
    cudaError_t e = cudaMemsetAsync(h->count_dev, 0, sizeof(unsigned), h->stream);
    if (e != cudaSuccess) return e;
    launch_count(h->P, h->tiles_pure, h->n_pure, h->pres[h->pp], h->count_dev, h->stream);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return cudaMemcpyAsync(h->count_host, h->count_dev, sizeof(unsigned), cudaMemcpyDeviceToHost, h->stream);
}

}  // namespace

extern "C" {

int lbm3_create(lbm3** out, const lbm3_grid* g, const uint8_t* solid, const double* angles,
                const double sigma[3], const double nu[3], double beta0, void* stream)
{
    if (!out) return fail(nullptr, LBM3_ERR_INVALID, "out is NULL");
    *out = nullptr;
    if (!g || !solid || !angles || !sigma || !nu)
        return fail(nullptr, LBM3_ERR_INVALID, "NULL argument");
    // the step kernel addresses the 27 population planes with 32-bit offsets
    if (g->nx < 8 || g->ny < 8 || 27LL * g->nx * g->ny >= (1LL << 31))
        return fail(nullptr, LBM3_ERR_INVALID, "grid must be at least 8x8 with 27 * nx * ny < 2^31");
    if (g->bc_x < 0 || g->bc_x > 3) return fail(nullptr, LBM3_ERR_INVALID, "bad bc_x");
    if (g->precision != LBM3_FP32 && g->precision != LBM3_FP16 && g->precision != LBM3_BF16)
        return fail(nullptr, LBM3_ERR_INVALID, "precision must be LBM3_FP32, LBM3_FP16 or LBM3_BF16");
    for (int j = 0; j < 3; j++) {
        if (!(sigma[j] > 0.0) || !std::isfinite(sigma[j]))
            return fail(nullptr, LBM3_ERR_INVALID, "sigma must be positive");
        if (!(nu[j] > 0.0) || !std::isfinite(nu[j]))
            return fail(nullptr, LBM3_ERR_INVALID, "nu must be positive");
    }
    if (!(beta0 >= 0.0)) return fail(nullptr, LBM3_ERR_INVALID, "beta0 must be >= 0");
    if (g->bc_x == kZouHe && (!(std::fabs(g->u_in) < 0.3) || !(g->rho_out > 0.0)))
        return fail(nullptr, LBM3_ERR_INVALID, "Zou-He needs |u_in| < 0.3 and rho_out > 0");
    if (g->bc_x == kModPer && sigma[0] != sigma[2])
        return fail(nullptr, LBM3_ERR_INVALID, "modified periodic boundary needs sigma_01 == sigma_12");

    const int nx = g->nx, ny = g->ny;
    const size_t N = (size_t)nx * ny;
    const Indicator S{nx, ny, g->periodic_y ? 1 : 0, g->bc_x, solid};

    // ---- node classes: a node is a boundary node when any D2Q9 neighbour is of the other kind
    std::vector<uint8_t> cls(N);
    // flags of the nodes: the directions that bounce back there, and the domain's edges
    std::vector<uint16_t> nflag(N);
    long long n_fluid = 0;
    for (int y = 0; y < ny; y++)
        for (int x = 0; x < nx; x++) {
            if (x == 1 && y > 0 && y < ny - 1) {
                const size_t row = (size_t)y * nx;
                n_fluid += classify_inside(solid + row, nx, cls.data() + row, nflag.data() + row);
                x = nx - 1;
            }
            const int me = S(x, y);
            bool touch = false;
            int flag = (x == 0 ? kNodeX0 : 0) | (x == nx - 1 ? kNodeXN : 0) | (y == 0 ? kNodeY0 : 0) |
                       (y == ny - 1 ? kNodeYN : 0);
            for (int a = 1; a < kQ; a++) {
                if (!me && S.outside_solid(x + ex(a), y + ey(a)))
                    return fail(nullptr, LBM3_ERR_INVALID,
                                "a fluid node touches a wall side: make the boundary rows/columns solid");
                const int other = S(x + ex(a), y + ey(a));
                if (other != me) touch = true;
                flag |= other << opp(a);
            }
            nflag[(size_t)y * nx + x] = (uint16_t)(me ? kNodeSolid : flag);
            cls[(size_t)y * nx + x] = me ? (touch ? kSB : kSI) : (touch ? kFB : kFI);
            n_fluid += !me;
        }
    if (g->bc_x == kZouHe) {
        if (!g->periodic_y) return fail(nullptr, LBM3_ERR_INVALID, "Zou-He boundary needs periodic y");
        for (int y = 0; y < ny; y++)
            for (int j = 0; j < 4; j++)
                if (solid[(size_t)y * nx + j] || solid[(size_t)y * nx + nx - 1 - j])
                    return fail(nullptr, LBM3_ERR_INVALID, "no solid node allowed within 4 columns of an open side");
    }

    // ---- wall list: C_SB nodes, outward normals by the eighth-order stencil, angle triples
    std::vector<int> widx;
    std::vector<double> wnrm;
    std::vector<float> wang;
    double young = 0.0;
    for (size_t i = 0; i < N; i++) {
        if (cls[i] != kSB) continue;
        const int x = (int)(i % nx), y = (int)(i / nx);
        double sx = 0.0, sy = 0.0;
        // eighth-order weights of Eq.(20) by |c|^2 (index = |c|^2)
        static const double w8[9] = {0.0, 4.0 / 21.0, 4.0 / 45.0, 0.0, 1.0 / 60.0, 2.0 / 315.0, 0.0, 0.0, 1.0 / 5040.0};
        for (int cy = -2; cy <= 2; cy++)
            for (int cx = -2; cx <= 2; cx++) {
                const int c2 = cx * cx + cy * cy;
                if (c2 == 0 || w8[c2] == 0.0) continue;
                if (S(x + cx, y + cy)) {
                    sx += w8[c2] * cx;
                    sy += w8[c2] * cy;
                }
            }
        double len = std::sqrt(sx * sx + sy * sy);
        if (len < 1e-12) {
            sx = sy = 0.0;
            for (int a = 1; a < kQ; a++)
                if (S(x + ex(a), y + ey(a))) {
                    const double w = a < 5 ? 1.0 / 9.0 : 1.0 / 36.0;
                    sx += w * ex(a);
                    sy += w * ey(a);
                }
            len = std::sqrt(sx * sx + sy * sy);
            if (len < 1e-12) {
                sx = 0.0;
                sy = -1.0;
                len = 1.0;
            }
        }
        widx.push_back((int)i);
        // Eq.(19) points into the solid; the characteristic lines leave along -n_s
        wnrm.push_back(-sx / len);
        wnrm.push_back(-sy / len);
        double th[3];
        for (int j = 0; j < 3; j++) {
            th[j] = angles[3 * i + j];
            if (!(th[j] > 0.0 && th[j] < 180.0))
                return fail(nullptr, LBM3_ERR_INVALID, "wall angles must lie in (0, 180) degrees");
            wang.push_back((float)th[j]);
        }
        const double d2r = M_PI / 180.0;
        const double r = sigma[0] * std::cos(th[0] * d2r) + sigma[1] * std::cos(th[1] * d2r) +
                         sigma[2] * std::cos(th[2] * d2r);
        young = std::max(young, std::fabs(r));
    }

    // ---- tiles of the fused step kernel (2-D prefix sums of the solid mask)
    std::vector<int> tp, tg, te;
    std::vector<int> rec;
    std::vector<int4> went;
    long long pure_fluid = 0;
    {
        std::vector<long long> ps((size_t)(nx + 1) * (ny + 1), 0);
        for (int y = 0; y < ny; y++)
            for (int x = 0; x < nx; x++)
                ps[(size_t)(y + 1) * (nx + 1) + x + 1] = ps[(size_t)y * (nx + 1) + x + 1] +
                                                         ps[(size_t)(y + 1) * (nx + 1) + x] -
                                                         ps[(size_t)y * (nx + 1) + x] +
                                                         (solid[(size_t)y * nx + x] ? 1 : 0);
        auto box = [&](int xa, int ya, int xb, int yb) {  // solids in [xa, xb) x [ya, yb)
            return ps[(size_t)yb * (nx + 1) + xb] - ps[(size_t)ya * (nx + 1) + xb] -
                   ps[(size_t)yb * (nx + 1) + xa] + ps[(size_t)ya * (nx + 1) + xa];
        };
        const int ntx = (nx + kTX - 1) / kTX, nty = (ny + kTY - 1) / kTY;
        for (int ty = 0; ty < nty; ty++)
            for (int tx = 0; tx < ntx; tx++) {
                const int x0 = tx * kTX, y0 = ty * kTY;
                const int x1 = std::min(nx, x0 + kTX), y1 = std::min(ny, y0 + kTY);
                // a tile without a fluid node has nothing to update (solid nodes are never
                // written and their populations never read): no block is launched for it
                if (box(x0, y0, x1, y1) == (long long)(x1 - x0) * (y1 - y0)) continue;
                const bool inner = x0 >= 3 && y0 >= 3 && x0 + kTX + 3 <= nx && y0 + kTY + 3 <= ny;
                if (inner && box(x0 - 3, y0 - 3, x0 + kTX + 3, y0 + kTY + 3) == 0) {
                    tp.push_back(ty * ntx + tx);
                    pure_fluid += (long long)kTX * kTY;
                } else if (inner) {
                    tg.push_back(ty * ntx + tx);
                } else {
                    te.push_back(ty * ntx + tx);
                }
            }
        // ---- the C_SB nodes that each of those wets, and the tiles whose stored fluids can reach it
        tg.insert(tg.end(), te.begin(), te.end());
        std::vector<int> wof(N, -1);
        for (size_t w = 0; w < widx.size(); w++) wof[widx[w]] = (int)w;
        std::vector<int> owner(widx.size(), -1);
        // tiles with a fluid node (the others are never written)
        std::vector<uint8_t> live((size_t)ntx * nty, 0);
        for (const int t : tp) live[t] = 1;
        for (const int t : tg) live[t] = 1;
        for (const int tile : tg) {
            const int x0 = (tile % ntx) * kTX, y0 = (tile / ntx) * kTY;
            const int first = (int)went.size();
            // columns and rows as the boundaries continue them: -1 where there is nothing
            constexpr int H = kNearHalo + 1;
            int col[kTX + 2 * H], par[kTX + 2 * H], row[kTY + 2 * H];
            bool open = false;
            for (int j = 0; j < kTX + 2 * H; j++) {
                int x = x0 + j - H;
                par[j] = 0;
                // a column that Zou-He completes may hold what nobody stored near it
                if (g->bc_x == kZouHe && (x <= 0 || x >= nx - 1)) open = true;
                if (x < 0 || x >= nx) {
                    if (g->bc_x == kZouHe || g->bc_x == kWalls) {
                        x = -1;
                    } else {
                        const int q = floordiv_i(x, nx);
                        x -= q * nx;
                        par[j] = g->bc_x == kModPer ? q & 1 : 0;
                    }
                }
                col[j] = x;
            }
            for (int j = 0; j < kTY + 2 * H; j++) {
                const int y = y0 + j - H;
                row[j] = y >= 0 && y < ny ? y : (g->periodic_y ? ((y % ny) + ny) % ny : -1);
            }
            std::vector<int> near, across;
            for (int j = 0; j < kTX + 2 * H; j++)
                if (col[j] >= 0) {
                    const int c = 2 * (col[j] / kTX) + par[j];
                    if (std::find(across.begin(), across.end(), c) == across.end()) across.push_back(c);
                }
            int seen = -1;
            for (int j = 0; j < kTY + 2 * H; j++) {
                if (row[j] < 0 || row[j] / kTY == seen) continue;
                seen = row[j] / kTY;
                for (const int c : across) {
                    const int t = seen * ntx + c / 2, code = 2 * t + (c & 1);
                    if (live[t] && std::find(near.begin(), near.end(), code) == near.end()) near.push_back(code);
                }
            }
            for (int cy = 0; cy < kTY + 4; cy++) {
                const int y = row[cy + H - 2];
                if (y < 0) continue;
                for (int cx = 0; cx < kTX + 4; cx++) {
                    const int x = col[cx + H - 2];
                    if (x < 0) continue;
                    const size_t i = (size_t)y * nx + x;
                    if (cls[i] != kSB) continue;
                    // the tile that has the node writes its wall values, else the first that sees it
                    const int w = wof[i], X = x0 + cx - 2, Y = y0 + cy - 2;
                    const bool mine = cx >= 2 && cx < kTX + 2 && cy >= 2 && cy < kTY + 2 && X < nx && Y < ny;
                    int own = 0;
                    if (mine || owner[w] < 0) {
                        if (owner[w] >= 0) went[owner[w]].z &= ~kWetOwner;
                        owner[w] = (int)went.size();
                        own = kWetOwner;
                    }
                    went.push_back(make_int4((int)i, w, cx | cy << 8 | (par[cx + H - 2] ? kWetPar : 0) | own, 0));
                }
            }
            if (open || (int)near.size() > kTileRecInts - kTileRecHead) near.assign(1, -1);
            near.resize(kTileRecInts - kTileRecHead, -2);
            rec.insert(rec.end(), {tile, first, (int)went.size() - first});
            rec.insert(rec.end(), near.begin(), near.end());
        }
    }
    const int n_gen = (int)tg.size();
    const char* chain_env = std::getenv("LBM3_CHAIN_TILES");
    const bool chain = n_gen + (int)tp.size() <= (chain_env ? std::atoi(chain_env) : kChainTiles);
    if (chain) {
        // a pure tile's record: no C_SB node, the 3 x 3 tiles around (it is inner, so they exist)
        const int ntx = (nx + kTX - 1) / kTX;
        for (const int t : tp) {
            rec.insert(rec.end(), {t, 0, 0});
            for (int m = 0; m < kTileRecInts - kTileRecHead; m++)
                rec.push_back(m < 9 ? 2 * (t + (m / 3 - 1) * ntx + m % 3 - 1) : -2);
        }
    }

    // ---- parameters
    lbm3* h = new lbm3();
    h->stream = (cudaStream_t)stream;
    h->precision = g->precision;
    Params& P = h->P;
    P.nx = nx;
    P.ny = ny;
    P.N = (long long)N;
    P.per_y = g->periodic_y ? 1 : 0;
    P.bc_x = g->bc_x;
    P.u_in = (float)g->u_in;
    P.rho_out = (float)g->rho_out;
    P.sig01 = (float)sigma[0];
    P.sig02 = (float)sigma[1];
    P.sig12 = (float)sigma[2];
    P.inv_nu0 = (float)(1.0 / nu[0]);
    P.inv_nu1 = (float)(1.0 / nu[1]);
    P.inv_nu2 = (float)(1.0 / nu[2]);
    P.beta0 = (float)beta0;
    // X_kl = (sigma_mk^2 + sigma_ml^2 - sigma_kl^2) / (2 sigma_mk sigma_ml), m = the third fluid
    const double s01 = sigma[0], s02 = sigma[1], s12 = sigma[2];
    P.g01 = (float)seg_g((s02 * s02 + s12 * s12 - s01 * s01) / (2.0 * s02 * s12));
    P.g02 = (float)seg_g((s01 * s01 + s12 * s12 - s02 * s02) / (2.0 * s01 * s12));
    P.g12 = (float)seg_g((s01 * s01 + s02 * s02 - s12 * s12) / (2.0 * s01 * s02));
    for (int k = 0; k < kNF; k++)
        for (int a = 0; a < kQ; a++) {
            P.off_plane[k * kQ + a] = (k * kQ + a) * (int)N;
            P.off_pull[k * kQ + a] = (k * kQ + a) * (int)N - ex(a) - ey(a) * nx;
            P.off_pull16[k * kQ + a] = k * (int)N - ex(a) - ey(a) * nx;
            P.off_pull16o[k * kQ + a] = a > 0 ? (8 * k + a - 1) * (int)N - ex(a) - ey(a) * nx : 0;
        }
    h->nw = (int)widx.size();
    h->n_fluid = n_fluid;
    h->n_pure = (int)tp.size();
    h->n_gen = n_gen;
    h->chain = chain;
    h->n_went = (int)went.size();
    h->pure_fluid = pure_fluid;
    h->wall_host = widx;

    // ---- device buffers
    auto dmalloc = [&](void** p, size_t b) -> cudaError_t {
        cudaError_t e = cudaMalloc(p, b ? b : 16);
        if (e == cudaSuccess) tally(h, b);
        return e;
    };
    cudaError_t e = cudaSuccess;
    for (int b = 0; b < 2; b++) {
        if (g->precision == LBM3_FP32) {
            if (e == cudaSuccess) e = dmalloc((void**)&h->pop[b].f, (size_t)27 * N * sizeof(float));
        } else {
            if (e == cudaSuccess) e = dmalloc((void**)&h->pop[b].rho, (size_t)3 * N * sizeof(float));
            if (e == cudaSuccess) e = dmalloc((void**)&h->pop[b].off, (size_t)24 * N * sizeof(unsigned short));
        }
    }
    if (e == cudaSuccess) e = dmalloc((void**)&h->type, N);
    for (int b = 0; b < 2; b++)
        if (e == cudaSuccess) e = dmalloc((void**)&h->cw[b], 3 * N * sizeof(double));
    if (e == cudaSuccess) e = dmalloc((void**)&h->u, 2 * N * sizeof(float));
    if (e == cudaSuccess) e = dmalloc((void**)&h->scratch, 3 * N * sizeof(double));
    if (e == cudaSuccess) e = dmalloc((void**)&h->partials, (size_t)diag_blocks(P) * 8 * sizeof(double));
    if (e == cudaSuccess) e = dmalloc((void**)&h->dout, 8 * sizeof(double));
    if (e == cudaSuccess) e = dmalloc((void**)&h->err_flag, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(h->err_flag, 0, sizeof(int));
    P.err = h->err_flag;
    P.wait_polls = kCopyWaitPolls;
    if (e == cudaSuccess) e = dmalloc((void**)&h->widx, widx.size() * sizeof(int));
    if (e == cudaSuccess) e = dmalloc((void**)&h->wnrm, wnrm.size() * sizeof(double));
    if (e == cudaSuccess) e = dmalloc((void**)&h->wang, wang.size() * sizeof(float));
    WetLane* cache = nullptr;
    if (e == cudaSuccess) e = dmalloc((void**)&cache, 4 * (size_t)h->n_went * sizeof(WetLane));
    h->gen.cache = cache;
    {
        std::vector<double2> en;
        for (const int4& w : went) en.push_back(make_double2(wnrm[2 * w.y], wnrm[2 * w.y + 1]));
        const void* from[5] = {rec.data(), went.data(), nflag.data(), tp.data(), en.data()};
        const size_t size[5] = {rec.size() * sizeof(int), went.size() * sizeof(int4), nflag.size() * sizeof(uint16_t),
                                tp.size() * sizeof(int), en.size() * sizeof(double2)};
        for (int j = 0; j < 5; j++) {
            if (e == cudaSuccess) e = dmalloc(&h->tile_mem[j], size[j]);
            if (e == cudaSuccess && size[j]) e = cudaMemcpy(h->tile_mem[j], from[j], size[j], cudaMemcpyHostToDevice);
        }
    }
    h->pres_bytes = (size_t)((nx + kTX - 1) / kTX) * ((ny + kTY - 1) / kTY) * sizeof(uint64_t);
    for (int b = 0; b < 2; b++) {
        if (e == cudaSuccess) e = dmalloc((void**)&h->pres[b], h->pres_bytes);
        if (e == cudaSuccess) e = cudaMemset(h->pres[b], 0x07, h->pres_bytes);
    }
    if (e == cudaSuccess) {
        int lo = 0, hi = 0;
        e = cudaDeviceGetStreamPriorityRange(&lo, &hi);
        if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&h->side, cudaStreamNonBlocking, hi);
        if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&h->side3, cudaStreamNonBlocking, hi);
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&h->gcap, cudaStreamNonBlocking);
    }
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ev_join3, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaMemcpy(h->type, cls.data(), N, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !widx.empty()) e = cudaMemcpy(h->widx, widx.data(), widx.size() * sizeof(int), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !wnrm.empty()) e = cudaMemcpy(h->wnrm, wnrm.data(), wnrm.size() * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !wang.empty()) e = cudaMemcpy(h->wang, wang.data(), wang.size() * sizeof(float), cudaMemcpyHostToDevice);
    for (int b = 0; b < 2; b++)
        if (e == cudaSuccess) e = cudaMemset(h->cw[b], 0, 3 * N * sizeof(double));
    if (e == cudaSuccess) e = cudaMemset(h->u, 0, 2 * N * sizeof(float));
    const char* one_env = std::getenv("LBM3_ONE_TILES");
    h->one = h->n_pure >= std::max(1, one_env ? std::atoi(one_env) : kOneTiles);
    // pure tiles through bulk tensor copies where the layout allows them (row pitch a multiple of
    // 16 bytes: nx % 4 == 0 for FP32 populations, nx % 8 == 0 for 16-bit offset planes);
    // LBM3_DISABLE_TMA=1 in the environment keeps the plain kernel
    if (e == cudaSuccess && nx % (g->precision == LBM3_FP32 ? 4 : 8) == 0 && h->n_pure > 0) {
        const char* off = std::getenv("LBM3_DISABLE_TMA");
        const bool f32 = g->precision == LBM3_FP32;
        bool maps = !(off && off[0] == '1');
        for (int b = 0; b < 2 && maps; b++)
            maps = f32 ? make_tensor_maps(P, h->pop[b].f, &h->tm_in_a[b], &h->tm_in_b[b], &h->tm_out[b])
                       : make_tensor_maps16(P, h->pop[b], &h->tm_in_a[b], &h->tm_in_b[b]);
        if (maps) {
            int dev = 0, sms = 0;
            e = cudaGetDevice(&dev);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            // a kernel that cannot get the shared memory it needs leaves the pure tiles on the plain
            // kernel (the same results), as when the tensor maps cannot be encoded
            cudaError_t ep = cudaSuccess;
            if (e == cudaSuccess) {
                ep = f32 ? step_tma_prepare() : step_tma16_prepare();
                if (ep != cudaSuccess) cudaGetLastError();
            }
            h->tma = e == cudaSuccess && ep == cudaSuccess && sms > 0;
            // FP32: the warp-specialised ring kernel, unless LBM3_PURE_KERNEL=tma asks for the
            // two-blocks-per-SM kernel (both give the same results)
            const char* pk = std::getenv("LBM3_PURE_KERNEL");
            if (h->tma && f32 && !(pk && std::strcmp(pk, "tma") == 0)) {
                bool rm = true;
                for (int b = 0; b < 2 && rm; b++) rm = make_box_map(P, h->pop[b].f, &h->tm_box[b]);
                h->ring = rm && step_ring_prepare() == cudaSuccess;
                if (!h->ring) cudaGetLastError();
            }
            // the two-blocks-per-SM kernel takes every pure tile itself
            if (h->tma && f32 && !h->ring) h->one = false;
            if (e == cudaSuccess) e = choose_blocks(h, sms);
        }
    }
    h->gen = TileSet{n_gen, (const int*)h->tile_mem[0], (const int4*)h->tile_mem[1], (const double2*)h->tile_mem[4], h->wang, h->gen.cache,
                     h->type, (const uint16_t*)h->tile_mem[2]};
    h->tiles_pure = (const int*)h->tile_mem[3];
    if (e != cudaSuccess) {
        const int code = e == cudaErrorMemoryAllocation ? LBM3_ERR_OOM : LBM3_ERR_CUDA;
        release(h);
        delete h;
        return fail(nullptr, code, std::string("device set-up failed: ") + cudaGetErrorString(e));
    }
    *out = h;
    if (young > 1e-6) {
        char buf[160];
        std::snprintf(buf, sizeof buf, "wall angles violate Eq.(18): max |sum sigma cos theta| = %.3g", young);
        h->err = buf;
        return LBM3_WARN_YOUNG;
    }
    h->err.clear();
    return LBM3_OK;
}

int lbm3_set_fields(lbm3* h, const double* rho)
{
    if (!h || !rho) return fail(h, LBM3_ERR_INVALID, "NULL argument");
    const size_t N = (size_t)h->P.N;
    double* drho = nullptr;
    CUDA_TRY(h, cudaMallocAsync((void**)&drho, 3 * N * sizeof(double), h->stream));
    CUDA_TRY(h, cudaMemcpyAsync(drho, rho, 3 * N * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    h->cur = 0;
    CUDA_TRY(h, pres_reset(h));
    CUDA_TRY(h, cudaMemsetAsync(h->err_flag, 0, sizeof(int), h->stream));
    launch_init(h->precision, h->P, drho, h->type, h->pop[0], h->stream);
    launch_wet_init(h->precision, h->P, h->nw, h->widx, h->pop[0], h->type, h->cw[h->pp], h->stream);
    launch_wet_look(h->P, h->gen, h->n_went, h->cw[h->pp], h->stream);
    CUDA_TRY(h, cudaMemsetAsync(h->u, 0, 2 * N * sizeof(float), h->stream));
    CUDA_TRY(h, cudaFreeAsync(drho, h->stream));
    CUDA_TRY(h, cudaGetLastError());
    h->ready = true;
    return LBM3_OK;
}

int lbm3_step(lbm3* h, int32_t nsteps)
{
    if (!h) return fail(h, LBM3_ERR_INVALID, "NULL handle");
    if (nsteps < 0) return fail(h, LBM3_ERR_INVALID, "nsteps < 0");
    if (!h->ready) return fail(h, LBM3_ERR_STATE, "lbm3_set_fields has not been called");
    // blocks of kGraphSteps steps through the graphs while at least one step remains after them;
    // the rest, and the last step (it writes the velocity), one by one
    int s = 0;
    for (; s + kGraphSteps < nsteps; s += kGraphSteps) {
        CUDA_TRY(h, count_tiles(h, kGraphSteps));
        CUDA_TRY(h, graph_block(h));
    }
    CUDA_TRY(h, count_tiles(h, nsteps - s));
    for (; s < nsteps; s++) CUDA_TRY(h, enqueue_step(h, s == nsteps - 1, nullptr));
    return LBM3_OK;
}

int lbm3_step_timed_detail(lbm3* h, int32_t nsteps, double ms_out[5])
{
    if (!h || !ms_out) return fail(h, LBM3_ERR_INVALID, "NULL argument");
    if (nsteps < 0) return fail(h, LBM3_ERR_INVALID, "nsteps < 0");
    if (!h->ready) return fail(h, LBM3_ERR_STATE, "lbm3_set_fields has not been called");
    for (int j = 0; j < 5; j++) ms_out[j] = 0.0;
    // The run's begin and end, and four a step around its launches -- none where a step is one launch,
    // which begins under the end of the one before as long as no event stands between them.
    const bool whole = chained(h);
    std::vector<cudaEvent_t> ev(2 + (whole ? 0 : 4 * (size_t)nsteps));
    for (auto& e : ev) CUDA_TRY(h, cudaEventCreate(&e));
    const cudaEvent_t begin = ev[0], end = ev[1];
    auto step_events = [&](int s) { return whole ? nullptr : &ev[2 + 4 * (size_t)s]; };
    // The steps are captured into one graph with the events as record nodes, so that they run
    // as lbm3_step runs them (replayed graphs) rather than launched one by one; launched one by
    // one if the capture fails.
    bool ran = false;
    if (nsteps > 0 && !h->graph_off) {
        const int c0 = h->cur, p0 = h->pp;
        cudaStream_t user = h->stream;
        h->stream = h->gcap;
        h->ev_external = true;
        cudaGraph_t g = nullptr;
        cudaGraphExec_t x = nullptr;
        cudaError_t ec = cudaStreamBeginCapture(h->gcap, cudaStreamCaptureModeThreadLocal);
        if (ec == cudaSuccess) {
            cudaError_t el = cudaEventRecordWithFlags(begin, h->gcap, cudaEventRecordExternal);
            for (int s = 0; s < nsteps && el == cudaSuccess; s++) el = enqueue_step(h, s == nsteps - 1, step_events(s));
            if (el == cudaSuccess) el = cudaEventRecordWithFlags(end, h->gcap, cudaEventRecordExternal);
            ec = cudaStreamEndCapture(h->gcap, &g);
            if (el != cudaSuccess) ec = el;
        }
        h->ev_external = false;
        h->stream = user;
        if (ec == cudaSuccess) ec = cudaGraphInstantiate(&x, g, 0);
        if (g) cudaGraphDestroy(g);
        if (ec == cudaSuccess) {
            // cur and pp turned during the capture as the steps turn them
            cudaError_t er = cudaGraphLaunch(x, h->stream);
            if (er == cudaSuccess) er = cudaStreamSynchronize(h->stream);
            cudaGraphExecDestroy(x);
            CUDA_TRY(h, er);
            ran = true;
        } else {
            h->cur = c0;
            h->pp = p0;
            cudaGetLastError();  // a failed capture leaves no sticky error; clear the last one
        }
    }
    if (!ran) {
        CUDA_TRY(h, cudaEventRecord(begin, h->stream));
        for (int s = 0; s < nsteps; s++) CUDA_TRY(h, enqueue_step(h, s == nsteps - 1, step_events(s)));
        CUDA_TRY(h, cudaEventRecord(end, h->stream));  // after the last step's joins
        CUDA_TRY(h, cudaStreamSynchronize(h->stream));
    }
    auto add = [&](int j, cudaEvent_t a, cudaEvent_t b) {
        float t = 0.f;
        const cudaError_t e = cudaEventElapsedTime(&t, a, b);
        ms_out[j] += t;
        return e;
    };
    if (nsteps > 0) CUDA_TRY(h, add(4, begin, end));
    if (whole) ms_out[2] = ms_out[4];
    for (int s = 0; s < nsteps && !whole; s++) {
        const cudaEvent_t* E = step_events(s);
        CUDA_TRY(h, add(1, E[0], E[1]));
        CUDA_TRY(h, add(2, E[2], E[3]));
    }
    for (auto& e : ev) cudaEventDestroy(e);
    return LBM3_OK;
}

int lbm3_step_timed(lbm3* h, int32_t nsteps, double ms_out[3])
{
    if (!ms_out) return fail(h, LBM3_ERR_INVALID, "NULL argument");
    double d[5];
    const int rc = lbm3_step_timed_detail(h, nsteps, d);
    if (rc != LBM3_OK) return rc;
    ms_out[0] = d[0];
    ms_out[1] = d[1];
    ms_out[2] = d[2] + d[3];
    return LBM3_OK;
}

int lbm3_fields(lbm3* h, double* rho_out, double* u_out)
{
    if (!h || !rho_out) return fail(h, LBM3_ERR_INVALID, "NULL argument");
    if (!h->ready) return fail(h, LBM3_ERR_STATE, "lbm3_set_fields has not been called");
    const size_t N = (size_t)h->P.N;
    launch_fields(h->precision, h->P, h->pop[h->cur], h->type, h->scratch, h->stream);
    CUDA_TRY(h, cudaGetLastError());
    touch_pages(rho_out, 3 * N);
    if (u_out) touch_pages(u_out, 2 * N);
    CUDA_TRY(h, cudaMemcpyAsync(rho_out, h->scratch, 3 * N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    if (u_out) {
        launch_widen(2 * N, h->u, h->scratch, h->stream);
        CUDA_TRY(h, cudaGetLastError());
        CUDA_TRY(h, cudaMemcpyAsync(u_out, h->scratch, 2 * N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    }
    return take_kernel_error(h);
}

int lbm3_diag(lbm3* h, double out[8])
{
    if (!h || !out) return fail(h, LBM3_ERR_INVALID, "NULL argument");
    if (!h->ready) return fail(h, LBM3_ERR_STATE, "lbm3_set_fields has not been called");
    launch_diag(h->precision, h->P, h->pop[h->cur], h->type, h->u, h->partials, h->dout, h->stream);
    CUDA_TRY(h, cudaGetLastError());
    CUDA_TRY(h, cudaMemcpyAsync(out, h->dout, 8 * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    if (int rc = take_kernel_error(h)) return rc;
    if (out[7] > 0.0 || !(out[6] > 0.0)) return fail(h, LBM3_ERR_DIVERGED, "non-finite or non-positive density");
    return LBM3_OK;
}

int lbm3_n_wall(const lbm3* h) { return h ? h->nw : LBM3_ERR_INVALID; }

int lbm3_wall_nodes(const lbm3* h, int32_t* idx, int32_t cap)
{
    if (!h || (!idx && cap > 0)) return LBM3_ERR_INVALID;
    const int n = std::min<int>(cap, h->nw);
    for (int j = 0; j < n; j++) idx[j] = h->wall_host[j];
    return h->nw;
}

int lbm3_wall_values(lbm3* h, double* c, int32_t cap)
{
    if (!h || (!c && cap > 0)) return fail(h, LBM3_ERR_INVALID, "NULL argument");
    if (!h->ready) return fail(h, LBM3_ERR_STATE, "lbm3_set_fields has not been called");
    const size_t N = (size_t)h->P.N;
    std::vector<double> cw(3 * N);
    CUDA_TRY(h, cudaMemcpyAsync(cw.data(), h->cw[h->pp], 3 * N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    CUDA_TRY(h, cudaStreamSynchronize(h->stream));
    const int n = std::min<int>(cap, h->nw);
    for (int j = 0; j < n; j++) {
        const size_t i = (size_t)h->wall_host[j];
        for (int k = 0; k < 3; k++) c[3 * j + k] = cw[k * N + i];
    }
    return h->nw;
}

int lbm3_get_state(lbm3* h, double* f_post, double* wall_c)
{
    if (!h || !f_post) return fail(h, LBM3_ERR_INVALID, "NULL argument");
    if (!h->ready) return fail(h, LBM3_ERR_STATE, "lbm3_set_fields has not been called");
    const size_t N = (size_t)h->P.N;
    float* post = nullptr;
    CUDA_TRY(h, cudaMallocAsync((void**)&post, 27 * N * sizeof(float), h->stream));
    launch_get_state(h->precision, h->P, h->pop[h->cur], h->type, post, h->stream);
    CUDA_TRY(h, cudaGetLastError());
    std::vector<float> tmp(27 * N);
    CUDA_TRY(h, cudaMemcpyAsync(tmp.data(), post, 27 * N * sizeof(float), cudaMemcpyDeviceToHost, h->stream));
    CUDA_TRY(h, cudaFreeAsync(post, h->stream));
    std::vector<double> cw;
    if (wall_c) {
        cw.resize(3 * N);
        CUDA_TRY(h, cudaMemcpyAsync(cw.data(), h->cw[h->pp], 3 * N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    }
    CUDA_TRY(h, cudaStreamSynchronize(h->stream));
    for (size_t i = 0; i < 27 * N; i++) f_post[i] = tmp[i];
    if (wall_c) std::memcpy(wall_c, cw.data(), 3 * N * sizeof(double));
    return LBM3_OK;
}

int lbm3_set_state(lbm3* h, const double* f_post, const double* wall_c)
{
    if (!h || !f_post || !wall_c) return fail(h, LBM3_ERR_INVALID, "NULL argument");
    const size_t N = (size_t)h->P.N;
    double* dpost = nullptr;
    CUDA_TRY(h, cudaMallocAsync((void**)&dpost, 27 * N * sizeof(double), h->stream));
    CUDA_TRY(h, cudaMemcpyAsync(dpost, f_post, 27 * N * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    h->cur = 0;
    CUDA_TRY(h, pres_reset(h));
    CUDA_TRY(h, cudaMemsetAsync(h->err_flag, 0, sizeof(int), h->stream));
    launch_set_state(h->precision, h->P, dpost, h->type, h->pop[0], h->stream);
    // both arrays: a step writes the C_SB nodes' values only (the second from the first: by way of the host
    // it made the call 8 % longer)
    CUDA_TRY(h, cudaMemcpyAsync(h->cw[0], wall_c, 3 * N * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    CUDA_TRY(h, cudaMemcpyAsync(h->cw[1], h->cw[0], 3 * N * sizeof(double), cudaMemcpyDeviceToDevice, h->stream));
    launch_wet_look(h->P, h->gen, h->n_went, h->cw[h->pp], h->stream);
    CUDA_TRY(h, cudaMemsetAsync(h->u, 0, 2 * N * sizeof(float), h->stream));
    CUDA_TRY(h, cudaFreeAsync(dpost, h->stream));
    CUDA_TRY(h, cudaGetLastError());
    CUDA_TRY(h, cudaStreamSynchronize(h->stream));
    h->ready = true;
    return LBM3_OK;
}

int lbm3_set_wall_angles(lbm3* h, const double* angles)
{
    if (!h || (!angles && h->nw > 0)) return fail(h, LBM3_ERR_INVALID, "NULL argument");
    std::vector<float> a(3 * (size_t)h->nw);
    for (size_t j = 0; j < a.size(); j++) {
        if (!(angles[j] > 0.0 && angles[j] < 180.0))
            return fail(h, LBM3_ERR_INVALID, "wall angles must lie in (0, 180) degrees");
        a[j] = (float)angles[j];
    }
    if (!a.empty())
        CUDA_TRY(h, cudaMemcpyAsync(h->wang, a.data(), a.size() * sizeof(float), cudaMemcpyHostToDevice, h->stream));
    // the lines that the next step reads were looked for with the old angles (and the words say that
    // they have settled)
    CUDA_TRY(h, pres_reset(h));
    if (h->ready) launch_wet_look(h->P, h->gen, h->n_went, h->cw[h->pp], h->stream);
    CUDA_TRY(h, cudaGetLastError());
    CUDA_TRY(h, cudaStreamSynchronize(h->stream));
    return LBM3_OK;
}

int lbm3_set_inflow(lbm3* h, double u_in)
{
    if (!h) return fail(h, LBM3_ERR_INVALID, "NULL handle");
    if (h->P.bc_x != kZouHe) return fail(h, LBM3_ERR_INVALID, "no Zou-He inlet");
    if (!(std::fabs(u_in) < 0.3)) return fail(h, LBM3_ERR_INVALID, "|u_in| must be < 0.3");
    if ((float)u_in == h->P.u_in) return LBM3_OK;  // the captured graphs stay valid
    h->P.u_in = (float)u_in;
    drop_graphs(h);  // the graphs hold the old Params
    return LBM3_OK;
}

int lbm3_adjoint_centroid(lbm3* h, int32_t nsteps, int32_t K, double* J_out, double* dJ_dangles,
                          double* dJ_du)
{
    if (!h || !J_out || !dJ_du || (!dJ_dangles && h->nw > 0)) return fail(h, LBM3_ERR_INVALID, "NULL argument");
    if (nsteps < 1 || K < 1) return fail(h, LBM3_ERR_INVALID, "nsteps and checkpoint_every must be >= 1");
    if (!h->ready) return fail(h, LBM3_ERR_STATE, "lbm3_set_fields has not been called");
    if (h->precision != LBM3_FP32) return fail(h, LBM3_ERR_INVALID, "the adjoint needs FP32 storage");
    if (h->P.bc_x == kModPer) return fail(h, LBM3_ERR_INVALID, "the adjoint does not support the modified periodic boundary");
    const size_t N = (size_t)h->P.N;
    const size_t fb = 27 * N * sizeof(float), cb = 3 * N * sizeof(double);
    const int nseg = (nsteps + K - 1) / K;
    const int seglen = std::min(K, nsteps);
    const int nck = std::max(nseg - 1, 1);
    lbm3::AdjStore& st = h->adj;
    cudaError_t e = cudaStreamSynchronize(h->stream);
    if (e == cudaSuccess && st.W && (st.nck < nck || st.nsg < seglen)) adj_release(h);
    if (e == cudaSuccess && !st.W) {
        if (e == cudaSuccess) e = cudaMalloc((void**)&st.ck_f, fb * nck);
        if (e == cudaSuccess) e = cudaMalloc((void**)&st.ck_c, cb * nck);
        if (e == cudaSuccess) e = cudaMalloc((void**)&st.sg_f, fb * seglen);
        if (e == cudaSuccess) e = cudaMalloc((void**)&st.sg_c, cb * seglen);
        if (e == cudaSuccess) e = cudaMalloc((void**)&st.fin_f, fb);
        if (e == cudaSuccess) e = cudaMalloc((void**)&st.fin_c, cb);
        // a step stores only the C_SB nodes' wall values into a state's slot; the rest
        // stays 0, as in the handle's own array
            if (e == cudaSuccess) e = cudaMemset(st.ck_c, 0, cb * nck);
        if (e == cudaSuccess) e = cudaMemset(st.sg_c, 0, cb * seglen);
        if (e == cudaSuccess) e = adjoint_alloc(h->P, h->nw, h->gen.nflag, &st.W);
        if (e == cudaSuccess && h->ring) {
            st.box.resize(seglen);
            for (int j = 0; j < seglen && e == cudaSuccess; j++)
                if (!make_box_map(h->P, st.sg_f + (size_t)j * 27 * N, &st.box[j])) e = cudaErrorInvalidValue;
        }
        st.nck = nck;
        st.nsg = seglen;
    }
    if (e != cudaSuccess) {
        adj_release(h);
        return fail(h, e == cudaErrorMemoryAllocation ? LBM3_ERR_OOM : LBM3_ERR_CUDA,
                    std::string("adjoint set-up: ") + cudaGetErrorString(e));
    }
    float *ck_f = st.ck_f, *sg_f = st.sg_f, *fin_f = st.fin_f;
    double *ck_c = st.ck_c, *sg_c = st.sg_c, *fin_c = st.fin_c;
    AdjointWork* W = st.W;
    auto cleanup = [&]() {
        if (e != cudaSuccess) adj_release(h);
    };
    cudaStream_t s = h->stream;
    // Where the step kernels can read any buffer (the ring path, through the slot's tensor map, the
    // plain kernels), a segment's steps go from slot to slot of the store.
    const bool direct = h->ring || !h->tma;
    // the current state into a slot of a store
    auto save = [&](float* df, double* dc) {
        cudaMemcpyAsync(df, h->pop[h->cur].f, fb, cudaMemcpyDeviceToDevice, s);
        cudaMemcpyAsync(dc, h->cw[h->pp], cb, cudaMemcpyDeviceToDevice, s);
    };
    auto slot = [&](int j) { return Pop{sg_f + (size_t)j * 27 * N, nullptr, nullptr}; };
    // one step from slot j to `out`, its wall values to cw_out
    auto slot_step = [&](int j, const Pop& out, double* cw_out, bool last) {
        const Pop in = slot(j);
        h->io_in = &in;
        h->io_out = &out;
        h->io_cw_out = cw_out;
        h->io_box = h->ring ? &st.box[j] : nullptr;
        const cudaError_t r = enqueue_step(h, last, nullptr);
        h->io_in = h->io_out = nullptr;
        h->io_cw_out = nullptr;
        h->io_box = nullptr;
        return r;
    };
    // n steps from slot 0 on, slot to slot
    auto slot_steps = [&](int n) {
        cudaError_t r = cudaSuccess;
        for (int j = 0; j < n && r == cudaSuccess; j++) r = slot_step(j, slot(j + 1), sg_c + (size_t)(j + 1) * 3 * N, false);
        return r;
    };
    // n steps of the handle's own buffers
    auto own_steps = [&](int n) {
        cudaError_t r = cudaSuccess;
        for (int j = 0; j < n && r == cudaSuccess; j++) r = enqueue_step(h, false, nullptr);
        return r;
    };
    auto restore = [&](const float* df, const double* dc) {
        h->cur = 0;
        pres_reset(h);
        cudaMemcpyAsync(h->pop[0].f, df, fb, cudaMemcpyDeviceToDevice, s);
        cudaMemcpyAsync(h->cw[0], dc, cb, cudaMemcpyDeviceToDevice, s);
        launch_wet_look(h->P, h->gen, h->n_went, h->cw[0], s);
    };
    // The whole sweep, enqueued without a host round trip (the seed reads J from the device
    // diagnostics): the forward pass with checkpoints, whose last segment's states go straight to
    // the segment store (with K >= nsteps: every state, no recompute at all), then the reverse
    // over the segments, each other segment recomputed from its checkpoint, then the final state
    // back into the handle.  capturing: recorded into a graph (no host waits allowed).
    auto enqueue_all = [&](bool capturing) -> cudaError_t {
        cudaError_t r = cudaSuccess;
        const int t_last = (nseg - 1) * K, n_last = nsteps - t_last;
        for (int seg = 0; seg < nseg - 1 && r == cudaSuccess; seg++) {
            save(ck_f + (size_t)seg * 27 * N, ck_c + (size_t)seg * 3 * N);
            r = own_steps(K);
        }
        if (r != cudaSuccess) return r;
        if (direct) {
            save(sg_f, sg_c);
            r = slot_steps(n_last - 1);
            // the final state in the handle's other buffer
            const int c = 1 - h->cur;
            if (r == cudaSuccess) r = slot_step(n_last - 1, h->pop[c], h->cw[c], true);
            h->cur = c;
            pres_reset(h);  // the words describe the slots, not the handle's buffers
        } else {
            for (int j = 0; j < n_last && r == cudaSuccess; j++) {
                save(sg_f + (size_t)j * 27 * N, sg_c + (size_t)j * 3 * N);
                r = enqueue_step(h, j == n_last - 1, nullptr);
            }
        }
        if (r != cudaSuccess) return r;
        launch_diag(h->precision, h->P, h->pop[h->cur], h->type, h->u, h->partials, h->dout, s);
        save(fin_f, fin_c);
        cudaMemsetAsync(adjoint_dang(W), 0, sizeof(double) * 3 * (size_t)std::max(h->nw, 1), s);
        cudaMemsetAsync(adjoint_du(W), 0, sizeof(double), s);
        adjoint_seed(h->P, W, h->pop[h->cur].f, h->type, h->dout, s);
        for (int seg = nseg - 1; seg >= 0 && r == cudaSuccess; seg--) {
            const int t0 = seg * K, t1 = std::min(nsteps, t0 + K);
            if (seg < nseg - 1 && direct) {
                // the checkpoint into slot 0, then slot to slot
                pres_reset(h);
                cudaMemcpyAsync(sg_f, ck_f + (size_t)seg * 27 * N, fb, cudaMemcpyDeviceToDevice, s);
                cudaMemcpyAsync(sg_c, ck_c + (size_t)seg * 3 * N, cb, cudaMemcpyDeviceToDevice, s);
                launch_wet_look(h->P, h->gen, h->n_went, sg_c, s);
                r = slot_steps(t1 - t0 - 1);
            } else if (seg < nseg - 1) {
                restore(ck_f + (size_t)seg * 27 * N, ck_c + (size_t)seg * 3 * N);
                for (int t = t0; t < t1 && r == cudaSuccess; t++) {
                    save(sg_f + (size_t)(t - t0) * 27 * N, sg_c + (size_t)(t - t0) * 3 * N);
                    if (t < t1 - 1) r = enqueue_step(h, false, nullptr);
                }
            }
            // the intermediates of step t - 1 are prepared on the adjoint's side stream while the
            // reverse of step t runs
            auto prepare = [&](int t, bool wait) {
                return adjoint_prepare(h->P, W, t, wait, h->nw, h->widx, h->wnrm, h->wang,
                                       sg_f + (size_t)(t - t0) * 27 * N, sg_c + (size_t)(t - t0) * 3 * N, h->type);
            };
            if (r == cudaSuccess) r = adjoint_sync(W, s);
            if (r == cudaSuccess) r = prepare(t1 - 1, false);
            for (int t = t1 - 1; t >= t0 && r == cudaSuccess; t--) {
                if (t > t0) r = prepare(t - 1, t + 1 < t1);
                if (r == cudaSuccess)
                    r = adjoint_reverse(h->P, W, t, h->nw, h->widx, h->wang, sg_c + (size_t)(t - t0) * 3 * N, h->type, s);
                if (r == cudaSuccess) r = cudaGetLastError();
            }
            // the segment's stored states are recomputed for the next segment; launched one by
            // one, the host waits for this segment's reverse before it enqueues that (running
            // further ahead made the sweep slower)
            if (r == cudaSuccess) r = adjoint_join(W, s);
            if (r == cudaSuccess && seg > 0 && !capturing) r = cudaStreamSynchronize(s);
        }
        restore(fin_f, fin_c);
        return r;
    };
    // Replayed as one CUDA graph, captured by the first call of a size (the graph holds the
    // store's addresses, so it lives as long as the store) and dropped with the handle's other
    // graphs when a captured parameter changes; launched one by one if the capture fails.
    if (st.gexec && (st.g_nsteps != nsteps || st.g_K != K || st.g_cur != h->cur)) {
        cudaGraphExecDestroy(st.gexec);
        st.gexec = nullptr;
    }
    if (!st.gexec && !h->graph_off) {
        const int cur0 = h->cur;
        cudaStream_t user = h->stream;
        h->stream = h->gcap;
        s = h->gcap;
        cudaGraph_t g = nullptr;
        cudaError_t ec = cudaStreamBeginCapture(h->gcap, cudaStreamCaptureModeThreadLocal);
        if (ec == cudaSuccess) {
            const cudaError_t el = enqueue_all(true);
            ec = cudaStreamEndCapture(h->gcap, &g);
            if (el != cudaSuccess) ec = el;
        }
        if (ec == cudaSuccess) ec = cudaGraphInstantiate(&st.gexec, g, 0);
        if (g) cudaGraphDestroy(g);
        h->stream = user;
        s = user;
        if (ec == cudaSuccess) {
            st.g_nsteps = nsteps;
            st.g_K = K;
            st.g_cur = cur0;
        } else {
            st.gexec = nullptr;
            cudaGetLastError();  // a failed capture leaves no sticky error; clear the last one
        }
        h->cur = cur0;  // the capture ran nothing
        h->pp = cur0;
    }
    if (st.gexec) {
        e = cudaGraphLaunch(st.gexec, s);
        h->cur = 0;  // where the sweep leaves the state (restore of the final state)
        h->pp = 0;
    } else {
        e = enqueue_all(false);
    }
    double d[8];
    std::vector<double> dang(3 * (size_t)std::max(h->nw, 1));
    double du = 0.0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(d, h->dout, sizeof d, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dang.data(), adjoint_dang(W), sizeof(double) * dang.size(), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&du, adjoint_du(W), sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cleanup();
    if (e != cudaSuccess) return fail(h, LBM3_ERR_CUDA, std::string("adjoint: ") + cudaGetErrorString(e));
    if (int rc = take_kernel_error(h)) return rc;
    *J_out = d[3] / d[0];
    for (int w = 0; w < h->nw; w++)
        for (int j = 0; j < 3; j++) dJ_dangles[3 * w + j] = dang[(size_t)j * h->nw + w];
    *dJ_du = h->P.bc_x == kZouHe ? du : 0.0;
    return LBM3_OK;
}

int lbm3_info(const lbm3* h, int64_t out[9])
{
    if (!h || !out) return LBM3_ERR_INVALID;
    for (int j = 0; j < 9; j++) out[j] = 0;
    out[0] = h->n_fluid;
    out[1] = h->nw;
    // populations read and written per fluid node: 27 FP32 (216 B), or per fluid an FP32 density
    // and 8 16-bit offsets (120 B); plus one class byte per node
    const long long per = h->precision == LBM3_FP32 ? 216 : 120;
    out[2] = h->n_fluid * per + h->P.N;
    out[3] = chained(h) ? 1 : (h->n_pure > 0) + 2 * h->one + (h->n_gen > 0);
    out[4] = 0;  // the wetting is part of the tiles' launch
    out[5] = (int64_t)h->bytes;
    // as if every node of the pure tiles held all three fluids
    out[6] = h->pure_fluid * per;
    out[7] = h->pure_fluid;
    out[8] = h->ring ? 2 : (h->tma ? 1 : 0);
    return LBM3_OK;
}

int lbm3_set_stream(lbm3* h, void* stream)
{
    if (!h) return LBM3_ERR_INVALID;
    const cudaStream_t next = (cudaStream_t)stream;
    if (next != h->stream) {
        // work already queued on the old stream (and the side stream, joined to it at the end of
        // every step) comes before anything later enqueued on the new one
        CUDA_TRY(h, cudaEventRecord(h->ev_fork, h->stream));
        CUDA_TRY(h, cudaStreamWaitEvent(next, h->ev_fork, 0));
    }
    h->stream = next;
    return LBM3_OK;
}

int lbm3_set_copy_wait_limit(lbm3* h, int32_t polls)
{
    if (!h) return LBM3_ERR_INVALID;
    h->P.wait_polls = polls < 0 ? kCopyWaitPolls : polls;
    drop_graphs(h);  // the graphs hold the old Params
    return LBM3_OK;
}

int lbm3_sync(lbm3* h)
{
    if (!h) return LBM3_ERR_INVALID;
    CUDA_TRY(h, cudaStreamSynchronize(h->stream));
    return LBM3_OK;
}

int lbm3_adjoint_release(lbm3* h)
{
    if (!h) return fail(h, LBM3_ERR_INVALID, "NULL handle");
    cudaError_t e = cudaStreamSynchronize(h->stream);
    adj_release(h);
    return e == cudaSuccess ? LBM3_OK : fail(h, LBM3_ERR_CUDA, std::string("adjoint release: ") + cudaGetErrorString(e));
}

void lbm3_destroy(lbm3* h)
{
    if (!h) return;
    cudaStreamSynchronize(h->stream);
    release(h);
    delete h;
}

const char* lbm3_last_error(const lbm3* h) { return h ? h->err.c_str() : g_create_error.c_str(); }

}  // extern "C"
