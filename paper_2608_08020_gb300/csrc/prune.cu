// The tournament's entry points (the kernel is in tournament.cu), the capacity of the
// tree, and gb_fork_slots: a tournament decided on another pool applied to this one.
#include "internal.cuh"

using namespace gb;

extern "C" gb_status gb_fork_slots(gb_pool* pool, const int32_t* parent_of_dev, gb_stream_t stream) {
  if (!pool || !parent_of_dev) return GB_ERR_INVALID;
  if (!pool->seeded) return fail(pool, GB_ERR_STATE, "pool not seeded");
  if (pool->next_layer != 0) return fail(pool, GB_ERR_STATE, "fork_slots inside an open step");
  if (pool->cfg.max_beams > kMaxBeams) return fail(pool, GB_ERR_UNSUPPORTED, "fork_slots: too many slots");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  prof_begin(pool, GB_PROF_PRUNE, s);
  // One launch: the forks and the shared-prefix segment rebuild that follows them.
  launch_forks(pool, parent_of_dev, s);
  gb_status st = check_launch(pool, "fork_slots");
  if (st != GB_OK) return st;
  prof_end(pool, GB_PROF_PRUNE, s);
  return GB_OK;
}

extern "C" gb_status gb_pool_set_capacity(gb_pool* pool, int capacity) {
  if (!pool) return GB_ERR_INVALID;
  if (capacity < 1 || capacity > pool->cfg.max_beams)
    return fail(pool, GB_ERR_INVALID, "set_capacity: 1 <= capacity <= max_beams required");
  pool->capacity = capacity;
  return GB_OK;
}

extern "C" gb_status gb_prune_branch(gb_pool* pool, int K, int fanout, int warmup, const uint8_t* eligible_dev,
                                     int32_t* parent_out_dev, uint8_t* pruned_out_dev, uint32_t* lineage_out_dev,
                                     gb_stream_t stream) {
  if (!pool) return GB_ERR_INVALID;
  if (K < 0 || fanout < 2) return fail(pool, GB_ERR_INVALID, "prune_branch: K >= 0 and fanout >= 2 required");
  if (!pool->seeded) return fail(pool, GB_ERR_STATE, "pool not seeded");
  if (pool->next_layer != 0) return fail(pool, GB_ERR_STATE, "prune_branch inside an open step");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  prof_begin(pool, GB_PROF_PRUNE, s);
  // One launch: the round and the shared-prefix segment rebuild that follows it.
  launch_prune_branch(pool, K, fanout, warmup, eligible_dev, parent_out_dev, pruned_out_dev, lineage_out_dev, s);
  gb_status st = check_launch(pool, "prune_branch");
  if (st != GB_OK) return st;
  prof_end(pool, GB_PROF_PRUNE, s);
  return GB_OK;
}
