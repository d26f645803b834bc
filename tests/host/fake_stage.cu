// fake_stage.cu -- the stage kernel's launches in the tests of the host code (fake_cuda.cpp): a
// line in the log, which for a batch compares the strips that each case's table counts with those
// in the list.
#include <map>
#include <string>

#include "lbfs_kernels.h"
#include "lbfs_stage.cuh"

extern "C" void fake_say(const char* what, cudaStream_t s, const char* more);

// What the cycles' kernel leaves behind when its grid barrier runs out: the mark, and a ticket of
// a residual that not every block has taken.
extern "C" void fake_cycles(void** args) {
    const lbfs::CycleArgs& a = *static_cast<const lbfs::CycleArgs*>(args[0]);
    const lbfs::PotCheck& ck = *static_cast<const lbfs::PotCheck*>(args[1]);
    a.cases[0].mg_tickets[1] = 7;
    ck.sync[1] = ck.sync[2] = 1;
}
// a residual: the ticket it finds
extern "C" void fake_residual(void** args, cudaStream_t s) {
    fake_say("ticket", s, std::to_string((*static_cast<const lbfs::DevCase**>(args[0]))->mg_tickets[1]).c_str());
}

namespace lbfs {

template <class R>
std::string misplaced(const StageCase<R>& c) {
    for (const void* p : {c.He[0], c.He[1], c.He[2], c.W[0], c.W[1], c.W[2], c.phi, c.Fs_prev, c.Sdot, c.mu})
        if (reinterpret_cast<size_t>(p) % 32) return " misplaced";
    return "";
}
template <class R, bool HALF, bool UNI>
cudaError_t stage_launch(const StageCase<R>& one, const StageCase<R>* cases, const TileRef* tiles, int ntiles, int, int,
                         cudaStream_t st) {
    std::map<int, int> n;
    for (int t = 0; t < ntiles; ++t) ++n[tiles[t].case_id];
    std::string more = UNI ? "one" + misplaced(one) : "batch";
    for (const auto& c : n)
        if (!UNI) more += misplaced(cases[c.first]);
    for (const auto& c : n)
        if (!UNI && cases[c.first].strips != c.second)
            more += " case " + std::to_string(c.first) + ": " + std::to_string(cases[c.first].strips) + " strips of " +
                    std::to_string(c.second);
    fake_say("stage", st, more.c_str());
    return cudaSuccess;
}
#define FAKE_STAGE(R, H, U) \
    template cudaError_t stage_launch<R, H, U>(const StageCase<R>&, const StageCase<R>*, const TileRef*, int, int, int, cudaStream_t);
FAKE_STAGE(float, true, true) FAKE_STAGE(float, false, true) FAKE_STAGE(float, true, false) FAKE_STAGE(float, false, false)
FAKE_STAGE(double, true, true) FAKE_STAGE(double, false, true) FAKE_STAGE(double, true, false) FAKE_STAGE(double, false, false)

}  // namespace lbfs
