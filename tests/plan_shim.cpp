// Host build of the rules that choose the form of a prefill or batch call (csrc/spmm_plan.h, csrc/spmspv_batch_form.h), for
// tests/test_spmm_pairs.py and tests/test_batch_form.py.  Compiled with g++ by the tests; not part of the library.
#include "spmm_plan.h"
#include "spmspv_batch_form.h"

extern "C" void shim_make_plan(long long R, long long nkb, long long N, int sms, int may_cut, long long* out) {
    const spdp::plan::Plan q = spdp::plan::make_plan(R, nkb, N, sms, may_cut != 0);
    const long long v[7] = {q.kernel, q.workers, q.rounds, q.sharers, q.slices, q.tiles, q.rest};
    for (int i = 0; i < 7; ++i) out[i] = v[i];
}
extern "C" int shim_pair_x_tiles(long long values_len, long long R, long long nkb) { return spdp::plan::pair_x_tiles(values_len, R, nkb); }
extern "C" int shim_batch_loads_one_by_one(long long nnz, long long uneven, long long M, long long K) {
    return spdp::plan::batch_loads_one_by_one(nnz, uneven, M, K);
}
