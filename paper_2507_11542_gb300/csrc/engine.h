// engine.h -- device-resident multi-instance stepping shared by the batched
// solve and the serving loop.
//
// An Engine owns one device arena (first-fit), a table of instance slots with
// their device descriptors (BatchInst), and per-group tile lists. Instances
// are admitted into free slots (arrays uploaded, CFL bound and non-finite
// check launched), activated together (one synchronisation: schedules and
// descriptors), advanced K RK3 steps at a time for all active instances (a
// captured CUDA graph replayed while the tile set is unchanged), and retired
// when their steps are done. Not thread-safe: one thread drives an Engine.
#pragma once

#include <cstdint>
#include <utility>
#include <vector>

#include "ctx.h"

namespace hj {

class Arena {
 public:
    void reset(unsigned char* base, size_t cap);
    bool alloc(size_t bytes, size_t* off);  // 256-byte aligned, first fit
    void release(size_t off, size_t bytes);
    size_t capacity() const { return cap_; }
    size_t used() const { return used_; }
    unsigned char* base() const { return base_; }

 private:
    unsigned char* base_ = nullptr;
    size_t cap_ = 0, used_ = 0;
    std::vector<std::pair<size_t, size_t>> free_;  // (offset, size), sorted by offset
};

struct Slot {
    bool used = false, active = false;
    hj_problem prob;                 // copy; slice_times points into `times`
    std::vector<double> times;
    void* out = nullptr;
    bool out_on_device = true;
    double* out_times = nullptr;
    GridDev G;
    int dtype = 0;
    size_t es = 0;
    long long N = 0;
    bool angles = false;
    int group = -1;
    int lane = 0;                    // rate class (Engine::init with lanes)
    int sx = 1, ty = 1, tz = 1;
    Schedule S;
    double sbi = 0.0;
    long long steps_total = 0, k_host = 0;
    size_t off = 0, bytes = 0;       // the slot's arena block
    size_t o_v = 0, o_v1 = 0, o_v2 = 0, o_td = 0, o_tf = 0, o_stage = 0, o_ends = 0, o_end_slice = 0, o_end_dt = 0;
    std::vector<double> table;       // host angle tables, alive until activation
    std::vector<float> table_f;
    hj_stats stats{};
    hj_status status = HJ_OK;
    uint64_t tag = 0;                // caller's identifier (problem index or ticket)
};

class Engine {
 public:
    ~Engine();
    // Allocates the arena (arena_bytes), descriptor table and reduction words.
    // With multirate, instances are sorted by size into rate lanes: per K
    // steps of the largest, smaller ones take kLaneMult[lane] * K (a server's
    // small requests do not wait for the pace of its largest ones). The lanes'
    // step blocks run concurrently, each on its own stream.
    hj_status init(hj_ctx* ctx, cudaStream_t stream, int max_slots, size_t arena_bytes, bool multirate = false);
    void shutdown();

    // Whether the batched row kernel serves this problem.
    static bool eligible(const hj_problem* p);
    // Arena bytes one problem needs.
    static size_t footprint(const hj_problem* p, bool out_on_device);

    int free_slot() const;
    // Copies the problem into a free slot and enqueues its upload, CFL bound
    // and non-finite check. HJ_EBUSY: no slot or arena space right now.
    hj_status admit(const hj_problem* p, void* out, bool out_on_device, double* out_times, uint64_t tag,
                    int* slot_out);
    // Activates every admitted slot: one synchronisation, then schedules,
    // launch shapes and descriptors. Slots whose v0 is not finite come back in
    // `failed` with status HJ_ENONFINITE and are released.
    hj_status activate(std::vector<int>* failed);
    // K RK3 steps of every active slot.
    hj_status run(int K);
    // How many steps to run next, `most` at most: no more than are left where a graph
    // has to be captured anyway (six steps of six 101^2 FP32 solves: 828 us of a
    // call with sixteen captured in two chains, 450 so).
    int block_steps(int most) const;
    bool any_active() const;
    // Active slots whose steps are all enqueued.
    void done_slots(std::vector<int>* out) const;
    // Finishes slots (duplicate slices, host copies, final checks), one
    // synchronisation; fills stats/out_times and releases them.
    hj_status retire(const std::vector<int>& slots);
    // Marks a slot finished now (cancellation) and releases it.
    hj_status drop(int slot);

    std::vector<Slot> slots;
    long long launches = 0;

 private:
    // Multipliers about inversely proportional to size, so that requests of
    // different sizes get similar shares of the GPU per tick (the smallest
    // lane's multiplier is capped: more steps of tiny launches only slow the
    // other lanes down). Chosen by measurement on the served workload.
    static constexpr int kLanes = 5;
    static constexpr int kLaneMult[kLanes] = {1, 2, 4, 8, 8};
    // lane of an instance of N nodes: the first l with N > kLaneNodes[l], else the last
    static constexpr long long kLaneNodes[kLanes - 1] = {1LL << 24, 1LL << 23, 1LL << 22, 1LL << 21};

    // The instances of a group are independent of each other, so a lane's share
    // of it is split into chains of launches that run concurrently (branches of
    // the step graph): one chain's last wave of blocks and its gaps between
    // launches are filled by another's. 24 solves of 2-D and 3-D grids (FP32):
    // 15.66 ms with all launches in one row, 15.30 with a chain a group, 15.10
    // with two, 15.8 with three, 16.3 with four.
    static constexpr int kChains = 2;
    struct Chain {
        size_t off = 0, end = 0;  // its tiles
    };
    struct Group {
        int dtype = 0, ndim = 0, dyn = 0, scheme = HJ_WENO5;
        int threads = 0, tz_target = 8;
        size_t smem = 0;
        std::vector<BatchTile> tiles;          // by lane, chain, then instance (largest first)
        std::vector<Chain> chains[kLanes];
        BatchTile* d_tiles = nullptr;
        size_t tile_cap = 0;
    };
    void deal(const std::vector<int>& members, std::vector<int>* part) const;
    std::vector<std::pair<int, int>> rank_shapes(const Group& g, const std::vector<int>& members);
    hj_status shape_group(Group& g, const std::vector<int>& members, const std::vector<int>& fresh);
    hj_status rebuild_tiles();
    // One RK3 step of a chain's instances.
    cudaError_t enqueue_step(const Group& g, const Chain& c, cudaStream_t s);
    // K steps of every chain of a lane, captured into a graph.
    cudaError_t capture_lane(int lane, int K, cudaGraph_t* graph);
    static int lane_of(long long nodes) {
        int l = 0;
        while (l < kLanes - 1 && nodes <= kLaneNodes[l]) ++l;
        return l;
    }
    long long dead_tiles() const;

    hj_ctx* ctx_ = nullptr;
    cudaStream_t stream_ = nullptr;
    cudaStream_t cap_stream_ = nullptr;          // capture only: the first chain
    std::vector<cudaStream_t> chain_stream_;     // capture and timing only: the others
    cudaEvent_t cap_ev_ = nullptr;
    int max_slots_ = 0;
    void* arena_mem_ = nullptr;
    Arena arena_;
    BatchInst* d_insts_ = nullptr;
    std::vector<BatchInst> h_insts_;
    unsigned long long* d_words_ = nullptr;  // per slot: CFL accumulator, non-finite flag
    std::vector<Group> groups_;
    bool tiles_dirty_ = true;
    long long tiles_total_ = 0;
    bool multirate_ = false;
    cudaGraphExec_t exec_[kLanes] = {};  // the step blocks of each lane
    int exec_K_[kLanes] = {};
    // multirate: each lane's step block runs on a stream of its own, forked
    // from and joined back into stream_, so that the lanes overlap on the GPU
    cudaStream_t lane_stream_[kLanes] = {};
    cudaEvent_t fork_ev_ = nullptr;
    cudaEvent_t lane_ev_[kLanes] = {};
    void drop_graphs();
    std::vector<int> pending_;
};

}  // namespace hj
