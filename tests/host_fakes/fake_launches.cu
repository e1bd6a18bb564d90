// The launchers of the library's other files, in their place: nothing runs, and the selection fails when a test says so.
#include "slaq_internal.cuh"

extern "C" {
int fake_fail_select = 0;          // selections from now on that cannot be launched
int fake_err_word = 0;             // what the next selection that reports finds in its handles' error words
}

namespace slaq {
int fit_prepare(slaq_handle*) { return 0; }
int select_setup(int* per_sm) { *per_sm = 1; return 0; }
int fit_least_lanes(const slaq_handle*) { return 2; }
int launch_fit(slaq_handle*, cudaStream_t, int) { return 1; }
int launch_gain(slaq_handle*, double, int, bool) { return 1; }
int launch_complete_gains(slaq_handle*) { return 1; }
static int selection(slaq_handle* const* hs, int n, uint32_t seq) {
    if (fake_fail_select > 0) return --fake_fail_select, -1;
    for (int s = 0; s < n; ++s) *hs[s]->err_word |= fake_err_word;
    if (seq) {
        hs[0]->mailbox->err = fake_err_word;
        hs[0]->mailbox->done = seq;
    }
    fake_err_word = 0;
    return 1;
}
int launch_select(slaq_handle* h, double, long long, int, bool, int32_t*, uint32_t seq) { return selection(&h, 1, seq); }
int launch_select_group(slaq_handle* const* hs, int n, double, long long, int, uint32_t seq, bool* whole) {
    *whole = true;
    return selection(hs, n, seq);
}
bool select_writes_whole_table(const slaq_handle*, long long) { return true; }
int launch_normalise_export(slaq_handle*, int32_t, const int64_t*, double*, double*, double*) { return 1; }
int launch_time_model(slaq_handle*, double*, double*) { return 1; }
int launch_shard_pick(slaq_handle*, int, long long) { return 1; }
int launch_shard_pass(slaq_handle*, int, int) { return 1; }
int launch_shard_count(slaq_handle*, int, const long long**) { return 1; }
int launch_shard_finalise(slaq_handle*, int, long long, const long long*, int32_t*) { return 1; }
}  // namespace slaq
