// art_internal.h -- host-side grid object shared by the translation units of the library.
#pragma once

#include <vector>

#include <cuda_runtime.h>

#include "art.h"
#include "art_device.cuh"

namespace art {

// A table in device memory that the host writes: what was last stored there, while that is known.
struct HostTable {
    std::vector<unsigned char> sent;
    bool known = false;
    bool in_graph = false;   // a graph holds a store to it
};

// What the device holds per source, once per direction: a forward trace and a reverse sweep need
// different luminosities, and alternating calls would replace each other's tables. One block of
// device memory.
struct SourceTables {
    SrcDev* src = nullptr;   // start of the block
    float* first = nullptr;  // forward: sums of first segments that do not fit behind the accumulator
    double* dL = nullptr;    // reverse: dloss/dL of callers that pass no buffer
    float* lum = nullptr;    // forward: base-ray non-ionizing luminosities; reverse: luminosities
    size_t cap = 0;          // sources
    size_t first_cap = 0;    // groups of 32 base rays
    HostTable src_sent, lum_sent, levels_sent;
};

}  // namespace art

struct art_grid {
    int device = 0;
    int sms = 1;
    cudaStream_t stream = nullptr;
    int n[3] = {0, 0, 0};
    long long ncell = 0;
    long long npad = 0;          // cells of the padded layout (sentinel ring around the grid)
    double lo[3] = {0, 0, 0};
    double dx = 1.0;
    int fbits = 0;               // fraction bits of the fixed-point distances
    const float* nH0 = nullptr;  // borrowed
    const float* nH = nullptr;   // borrowed, may be NULL
    std::vector<double> pos, L;  // host copies of the sources
    std::vector<double> Ln;      // non-ionizing luminosities (two-bin traces)
    bool two_bin = false;
    float2* d_chi2 = nullptr;    // {chi_i, chi_n} per cell length (two-bin traces, padded)
    std::vector<int> src_lmax;
    art::SourceTables tables[2];     // forward, reverse
    art::LevelInfo* d_levels = nullptr;  // level constants, kNL per direction
    std::vector<void*> retired;      // former blocks of the forward tables (see prepare_trace)
    bool first_ordered = false;      // the prepared trace keeps its first segments
    float* d_first = nullptr;        // where: behind the accumulator or in tables[0]
    size_t first_room = 0;           // float4s behind the accumulator (a 32nd of it)

    // device buffers owned by the grid
    float* d_chi = nullptr;      // opacity per cell length (padded layout)
    float4* d_acc = nullptr;     // per-cell accumulator (padded layout); traces without a force
                                 // and the reverse sweep's gradient use the first npad floats
    art::DevState* d_state = nullptr;  // scheduler and counters, cleared together
    bool state_clean = false;          // d_state is clear once the stream gets here
    bool state_dirty_captured = false; // this trace's clearing of it is only captured
    art::Sched* d_sched = nullptr;     // in d_state
    art::DevStats* d_stats = nullptr;  // in d_state
    art::DevStats* h_stats = nullptr;  // pinned

    float4* dir[art::kNL] = {};     // per level: 3 float4 per pixel (n as df, face spacing codes)
    bool dir_built[art::kNL] = {};
    bool dir_rotate = false;
    double dir_rot[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1};

    // forward fronts (quads) of the levels beyond l0
    art::QuadBuf quad[art::kNL] = {};
    unsigned long long quad_cap[art::kNL] = {};      // allocated quads per level

    // adjoint fronts
    art::AdjBuf adj[art::kNL] = {};
    unsigned long long adj_cap[art::kNL] = {};       // allocated quads per level

    // adjoint: cell records
    float4* d_rec = nullptr;     // per-cell {chi, chi_H, w, 0} of the reverse sweep (padded)
    art::CellF* d_recf = nullptr;  // the same with the force weight (loss with a force term)
    art::CellW* d_recw = nullptr;  // {chi, w} per cell (loss without dust or force term)

    int lmax_glob = 0;
    int last_lmax = 0;
    int last_kind = 0;  // 0 forward, 1 backward
    double last_L_in = 0.0;
    double last_Ln_in = 0.0;
    bool last_two_bin = false;
    unsigned long long destroy_expected = 0;
    bool traced = false;
};

namespace art {
int check_params(const art_params* p);
int ensure_directions(art_grid* g, const art_params* p, int lfrom, int lto);
int run_opacity(art_grid* g, const art_params* p, bool two_bin, bool clear4, bool clear1, DevStats* st);
int begin_trace(art_grid* g);
void end_trace(art_grid* g);
int trace_threads(const art_params* p);
int cell_blocks(long long n);
double rmax_cells(double m_ray, int level);
fix to_fix(double cells, int fbits);
Coef coef_of(double v);
SrcDev source_record(const art_grid* g, const double u[3], double base_L, int lmax);
int prepare_trace(art_grid* g, const art_params* p, bool adjoint);
TraceArgs make_args(art_grid* g, const art_params* p, bool adjoint);
int finish_stats(art_grid* g, art_stats* out);
}  // namespace art
