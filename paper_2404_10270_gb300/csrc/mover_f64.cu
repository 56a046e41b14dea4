// mover_f64.cu -- instantiations of the fused mover for double particle state.
#include "kernels.h"
#include "mover.cuh"

namespace bitpic {

namespace {
// One launch of a variant with the shared memory of its ring.
template <int NT, bool MAG, bool MOVE, bool SUB, bool MIXED, MoveMode MODE>
cudaError_t launch(const MoveArgs& a, int grid, cudaStream_t st)
{
    k_move<double, NT, MAG, MOVE, SUB, MIXED, MODE><<<grid, NT, ring_bytes<double, MODE>(NT), st>>>(a);
    return cudaGetLastError();
}

template <int NT, bool SUB, MoveMode MODE>
cudaError_t go_sub(const MoveArgs& a, bool mag, bool mixed, int grid, cudaStream_t st)
{
    if (!mag) return launch<NT, false, true, SUB, false, MODE>(a, grid, st);
    // (the Boris form loads directly, see k_move)
    constexpr MoveMode M = MODE == MoveMode::kAhead ? MoveMode::kDirect : MODE;
    return mixed ? launch<NT, true, true, SUB, true, M>(a, grid, st)
                 : launch<NT, true, true, SUB, false, M>(a, grid, st);
}

template <int NT, bool SUB>
cudaError_t go_mode(const MoveArgs& a, bool mag, bool mixed, MoveMode mode, int grid, cudaStream_t st)
{
    if (mode == MoveMode::kFull) return go_sub<NT, SUB, MoveMode::kFull>(a, mag, mixed, grid, st);
    if (mode == MoveMode::kAhead) return go_sub<NT, SUB, MoveMode::kAhead>(a, mag, mixed, grid, st);
    return go_sub<NT, SUB, MoveMode::kDirect>(a, mag, mixed, grid, st);
}

template <int NT>
cudaError_t go(const MoveArgs& a, bool mag, bool move, bool sub, bool mixed, bool sort,
               MoveMode mode, int grid, cudaStream_t st)
{
    if (!move) return launch<NT, false, false, false, false, MoveMode::kDirect>(a, grid, st);
    if (sort) return launch_sort_step<double, NT>(a, mag, sub, mixed, grid, st);
    return sub ? go_mode<NT, true>(a, mag, mixed, mode, grid, st)
               : go_mode<NT, false>(a, mag, mixed, mode, grid, st);
}

// Resident blocks per SM; also raises the variant's shared-memory limit (a block's rings
// pass 48 KB), outside any stream capture.
template <int NT, bool MAG, bool SUB, bool MIXED, MoveMode MODE>
int resident_one()
{
    const auto k = k_move<double, NT, MAG, true, SUB, MIXED, MODE>;
    const int sm = (int)ring_bytes<double, MODE>(NT);
    int n = 0;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, NT, sm);
    return e == cudaSuccess ? n : 0;
}
template <int NT, bool SUB, MoveMode MODE>
int resident(bool mag)
{
    if (!mag) return resident_one<NT, false, SUB, false, MODE>();
    // (the Boris form loads directly, see k_move)
    constexpr MoveMode M = MODE == MoveMode::kAhead ? MoveMode::kDirect : MODE;
    if (resident_one<NT, true, SUB, true, M>() == 0) return 0;
    return resident_one<NT, true, SUB, false, M>();
}
template <int NT, bool SUB>
int resident_mode(bool mag, MoveMode mode)
{
    if (mode == MoveMode::kFull) return resident<NT, SUB, MoveMode::kFull>(mag);
    if (mode == MoveMode::kAhead) return resident<NT, SUB, MoveMode::kAhead>(mag);
    return resident<NT, SUB, MoveMode::kDirect>(mag);
}

template <int NT>
int occupancy(bool mag, bool sub, bool sort, bool yp, MoveMode mode)
{
    if (sort) return sort_step_blocks_per_sm<double, NT>(mag, yp);
    return sub ? resident_mode<NT, true>(mag, mode) : resident_mode<NT, false>(mag, mode);
}
}  // namespace

cudaError_t launch_move_f64(const MoveArgs& a, bool mag, bool move, bool sub, bool mixed,
                            bool sort, MoveMode mode, int nt, int grid, cudaStream_t st)
{
    switch (nt) {
        case 128: return go<128>(a, mag, move, sub, mixed, sort, mode, grid, st);
        case 512: return go<512>(a, mag, move, sub, mixed, sort, mode, grid, st);
        default: return go<256>(a, mag, move, sub, mixed, sort, mode, grid, st);
    }
}

int move_blocks_per_sm_f64(bool mag, bool sub, bool sort, bool yp, MoveMode mode, int nt)
{
    switch (nt) {
        case 128: return occupancy<128>(mag, sub, sort, yp, mode);
        case 512: return occupancy<512>(mag, sub, sort, yp, mode);
        default: return occupancy<256>(mag, sub, sort, yp, mode);
    }
}

}  // namespace bitpic
