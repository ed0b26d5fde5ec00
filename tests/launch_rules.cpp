// The host-side launch rules of the kernels, for tests/test_launch_rules_host.py.
#include "kvt_internal.h"

extern "C" {
int64_t grid_ctas(int64_t items, int64_t cap) { return kvt::item_grid(items, cap); }
int64_t copy_threads() { return kvt::kCopyThreads; }
int32_t migration_ctas(int32_t limit, int32_t beside, int32_t sms) {
    return kvt::migration_ctas(limit, beside != 0, sms);
}
int64_t inline_blocks() { return kvt::kResumeInlineMax; }
}
