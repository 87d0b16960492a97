// The library's pair planning as plain functions for the tests: host work only, but for replan_one_sided.
#include "common.cuh"
#include "tree_host.hpp"

#include <cstring>

using namespace ctr;

namespace ctr {
int schedule_slots(int sms, int slots[3]);
}

namespace {
int64_t put(const std::vector<PairItem>& v, int64_t cap, int32_t* out) {   // {I, j_begin, j_end, kind} each
    if ((int64_t)v.size() <= cap) std::memcpy(out, v.data(), sizeof(PairItem) * v.size());
    return (int64_t)v.size();
}
}  // namespace

extern "C" {

int closed_fit(int64_t M, int64_t E) { return closed_lists_fit(M, E) ? 1 : 0; }

int64_t plan_direct(int64_t M, int BS, const uint8_t* flags, int g0, int nb0, int closed, int64_t cap, int32_t* out) {
    return put(direct_runs(M, BS, std::vector<uint8_t>(flags, flags + (size_t)nb0 * nb0), g0, nb0, closed != 0), cap, out);
}

// A direct schedule of M nodes without correction pairs cut into items: their number; pairs: one-sided and symmetric
int64_t cut_direct(int pol, int64_t M, int BS, int tile, int slots, int64_t* pairs, int64_t cap, int32_t* out) {
    const int nb = (int)((M + BS - 1) / BS);
    PairSchedule p;
    p.BS = BS;
    p.tile = tile;
    cut_runs(p, pol, M, direct_runs(M, BS, std::vector<uint8_t>((size_t)nb * nb, 0), BS, nb, true), slots);
    pairs[0] = p.pairs_one;
    pairs[1] = p.pairs_sym;
    return put(p.items, cap, out);
}

// ptr, excl: correction rows in tree positions; near ranges of every block as ctr_farfield_plan gives them
int64_t plan_tree(int64_t M, int BS, const int32_t* ptr, const int32_t* excl, int64_t nb, const int64_t* near_ptr,
                  const int32_t* near_rng, int closed, int64_t cap, int32_t* out) {
    tree::Lists L;
    L.BS = BS;
    L.near_ptr.assign(near_ptr, near_ptr + nb + 1);
    L.near_rng.assign(near_rng, near_rng + 2 * near_ptr[nb]);
    const std::vector<uint8_t> corr = correction_blocks(M, std::vector<int32_t>(ptr, ptr + M + 1),
                                                        std::vector<int32_t>(excl, excl + ptr[M]));
    return put(near_runs(L, M, BS, corr, closed != 0), cap, out);
}

// Plans a direct handle's schedules again as one whose closed exclusion lists do not fit.
int replan_one_sided(ctr_ibim* s) {
    int sms = 0, slots[3];
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, s->device) != cudaSuccess) return -1;
    s->closed = false;
    for (PairSchedule& p : s->sched) p.planned = false;
    const int st = schedule_slots(sms, slots);
    return st < 0 ? st : plan_schedules(s, slots);
}

// What the engine takes one application of arithmetic pol (0 FP32, 1 float-float, 2 FP64) to last
double estimated_seconds(const ctr_ibim* s, int pol) { return s->sched[pol].total_cost / kUnitRate[pol]; }
}
