// The host-side launch rules of the kernels, for tests/test_launch_rules_host.py.
#include "decode_launch.h"

extern "C" {
int64_t grid_ctas(int64_t items, int64_t cap) { return kvt::item_grid(items, cap); }
int64_t copy_threads() { return kvt::kCopyThreads; }
int32_t migration_ctas(int32_t limit, int32_t beside, int32_t sms) {
    return kvt::migration_ctas(limit, beside != 0, sms);
}
int64_t shared_part_rows(int64_t rows, int32_t sms, int32_t group) {
    return kvt::shared_part_rows(rows, sms, group);
}
// shape: sub, per_sm, pace, merge_max_splits, one_split, by_length, wide, combine
void decode_shape(int32_t max_blocks, int32_t bt, int32_t Hq, int32_t Hkv, int32_t layers, int32_t B,
                  int64_t part_rows, int32_t sms, int32_t overlap, int32_t *shape) {
    kvt::DecodeArgs a = {};
    a.max_blocks = max_blocks;
    a.nlayers = layers;
    a.B = B;
    a.part_rows = part_rows;
    a.s.Hq = Hq;
    a.s.Hkv = Hkv;
    a.s.bt = bt;
    const int splits = kvt::max_splits_for(static_cast<int64_t>(max_blocks) * bt);
    const kvt::DecodeShape d = kvt::decode_shape(a, splits, sms, overlap != 0);
    const int32_t v[8] = {d.sub, d.per_sm, d.pace, d.merge_max_splits,
                          d.one_split, d.by_length, d.wide, d.combine};
    for (int i = 0; i < 8; ++i) shape[i] = v[i];
}
int64_t inline_blocks() { return kvt::kResumeInlineMax; }
}
