// FP32 instantiation of the step kernels (deviation storage, FP64 reductions).
#include "enqueue.cuh"

namespace hgks {
HGKS_INSTANTIATE(float)

int march_share(const std::vector<Engine*>& members) {
  std::vector<long long> rows;
  for (const Engine* e : members) rows.push_back(march_args(*e, static_cast<const float*>(e->q)).start[3]);
  return march_share_of(rows, members[0]->sms);
}
}  // namespace hgks
