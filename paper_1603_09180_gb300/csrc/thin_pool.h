// thin_pool.h -- which memory pool a call's scratch comes from.  Host logic
// only: a host compiler can build it without CUDA.
#pragma once

namespace thin {

// The library's pool on one device.
template <typename Pool>
struct PoolSlot {
    unsigned long long ctx_id = 0;  // context the pool belongs to
    Pool pool = Pool();
};

// The pool for a call in the context `ctx_id` (0: none): the library's own in
// the device's primary context, which the CUDA runtime uses, and none (the
// device's default pool) in any other.  A pool per device is all there is, also
// where a program goes back and forth between contexts; another one is made
// only when the primary context has been created anew and the old pool went
// with it.  is_primary() and create(Pool *) are asked for no more than that.
template <typename Pool, typename IsPrimary, typename Create>
Pool pool_for(PoolSlot<Pool> &S, unsigned long long ctx_id, IsPrimary is_primary, Create create)
{
    if (ctx_id == 0) return Pool();
    if (S.pool && S.ctx_id == ctx_id) return S.pool;
    Pool made = Pool();
    if (!is_primary() || !create(&made)) return Pool();
    S.pool = made;
    S.ctx_id = ctx_id;
    return made;
}

}  // namespace thin
