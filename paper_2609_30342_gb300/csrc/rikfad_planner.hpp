// rikfad_planner.hpp -- host-side construction of the work plan (no CUDA).
#pragma once
#include <string>
#include <vector>

#include "rikfad.h"
#include "rikfad_plan.hpp"

namespace rikfad {

struct Plan {
    std::vector<TensorDev> tensors;
    std::vector<PanelDev> panels;
    std::vector<PieceDev> pieces;
    std::vector<int32_t> block_piece;   // block b owns pieces [block_piece[b], block_piece[b+1])
    std::vector<int64_t> slot_off;      // colpart offset of every slot
    std::vector<FinItemDev> fin_items;
    std::vector<TileGroupDev> tile_groups;   // every tensor, in memory order (build_tiles)
    int band_width = 0;                 // columns of the widest band (0: no bands)
    bool elements_only = false;         // no matrix has rows: the step is a pass over tiles
    int64_t fac_floats = 0;             // factors + element-wise friction (padded)
    int64_t rowpart_floats = 0;
    int64_t colpart_floats = 0;
    int32_t spart_floats = 0;
    int nblocks = 0;                    // blocks of the step kernel (0 when there is no work)
    int64_t total_bytes = 0;            // compulsory HBM bytes of one step (planner's cost model)

    // In-order schedule (see rikfad_plan.hpp)
    std::vector<UnitDev> units;
    std::vector<NodeDev> nodes;
    std::vector<PanelTreeDev> trees;    // one per panel
    int64_t partial_floats = 0;         // unit and node partials
};

// Add the in-order schedule (units, reduction trees) to a plan built by
// build_plan.  Matrices keep their order; vectors come last.
void build_sweep(const rikfad_shape *shapes, int ntensors, Plan &plan);

// Add the tiles of every tensor: rows before panels.  Their number grows with the
// elements (the rest of a plan with blocks, rows and columns), so that only a handle
// has them, once its factors are allocated, and a plan query none.  Returns "" or an
// error message.
std::string build_tiles(Plan &plan);

// Validate the shape list; returns "" or an error message.
std::string check_shapes(const rikfad_shape *shapes, int ntensors);

// The ragged rows of a list (cols % 8 != 0), which the step kernel updates in
// single elements.
RaggedKind ragged_kind(const rikfad_shape *shapes, int ntensors);

// Build the plan for at most max_blocks blocks.  grad_bytes is 2 or 4.
// Returns "" on success or an error message.
// full_matrices: every matrix keeps element-wise friction (m x n floats)
// and its R, C become shadow factors (full iKFAD with R-iKFAD's factors
// carried alongside).
std::string build_plan(const rikfad_shape *shapes, int ntensors, int grad_bytes, int max_blocks,
                       Plan &plan, bool full_matrices = false);

// Bytes of one step that HBM must move for one element (compulsory traffic):
// matrix element: read grad + X + P, write X + P; vector element: + friction
// read and write.
inline int64_t matrix_elem_bytes(int grad_bytes) { return grad_bytes + 16; }
inline int64_t vector_elem_bytes(int grad_bytes) { return grad_bytes + 24; }

// build_plan for as many blocks as a plan's own launch lets run at once:
// `resident(plan)` returns that number for a plan with bands, whose launch takes
// shared memory by its widest band (0: cannot run; the result is then an error).
// A plan for fewer blocks has larger shares and can so have wider bands: the
// plan returned is one that `resident` was asked about last.  max_blocks is
// lowered to what was planned for.
template <typename F>
std::string build_resident_plan(const rikfad_shape *shapes, int ntensors, int grad_bytes, int &max_blocks, Plan &plan,
                                bool full_matrices, F resident)
{
    for (;;) {
        const std::string err = build_plan(shapes, ntensors, grad_bytes, max_blocks, plan, full_matrices);
        if (!err.empty() || plan.band_width == 0)
            return err;
        const int fit = resident(plan);
        if (fit < 1)
            return "step kernel cannot be resident on this device";
        if (fit >= max_blocks)
            return "";
        max_blocks = fit;
    }
}

}  // namespace rikfad
