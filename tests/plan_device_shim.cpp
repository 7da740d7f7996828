// Host build of the rule that cuts a prefill call on a device with thread-block clusters (csrc/spmm_plan.h), for
// tests/test_spmm_device_plans.py.  Compiled with g++ by the test; not part of the library.
#include "spmm_plan.h"

extern "C" void shim_device_plan(long long R, long long nkb, long long N, int sms, const int* resident, long long* out) {
    const spdp::plan::Plan q = spdp::plan::make_plan(R, nkb, N, sms, true, resident);
    const long long v[8] = {q.kernel, q.workers, q.rounds, q.sharers, q.slices, q.tiles, q.rest, q.cluster};
    for (int i = 0; i < 8; ++i) out[i] = v[i];
}
extern "C" int shim_pair_acc_tokens(long long N) { return spdp::plan::pair_acc_tokens(N); }
extern "C" int shim_pair_tile_tokens(long long N) { return spdp::plan::pair_tile_tokens(N); }
extern "C" int shim_pair_tiles_in_flight(long long values_len, long long R, long long nkb) { return spdp::plan::pair_x_tiles(values_len, R, nkb); }
extern "C" void shim_device_plan_wide(long long R, long long nkb, long long N, int sms, const int* resident, long long* out) {
    const spdp::plan::Plan q = spdp::plan::make_plan(R, nkb, N, sms, true, resident, true);
    const long long v[9] = {q.kernel, q.workers, q.rounds, q.sharers, q.slices, q.tiles, q.rest, q.cluster, q.sets};
    for (int i = 0; i < 9; ++i) out[i] = v[i];
}
