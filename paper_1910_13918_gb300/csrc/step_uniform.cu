// The fused uniform step with FP32 storage (step_uniform.cuh); each storage type is a translation
// unit of its own so that they compile side by side.
#include "step_uniform.cuh"

namespace sllbm {

cudaError_t launch_step_uniform_bf16(const StepArgs& a, const UniformTables& t, cudaStream_t s);

cudaError_t launch_step_uniform(const StepArgs& a, const UniformTables& t, int store, cudaStream_t s) {
  if (store == kStoreBF16) return launch_step_uniform_bf16(a, t, s);
  return launch_step_uniform_store<float>(a, t, s);
}

void uniform_edge_tiles(int P, int nx, int ny, UniformTables& t, std::vector<int2>& tiles) {
  int r[4] = {0, 0, 0, 0}, ty = 8;
  switch (P) {
    case 1: interior_tiles<1>(nx, ny, t.px0, t.px1, t.py0, t.py1, r); ty = TileShape<1>::TY; break;
    case 2: interior_tiles<2>(nx, ny, t.px0, t.px1, t.py0, t.py1, r); ty = TileShape<2>::TY; break;
    case 3: interior_tiles<3>(nx, ny, t.px0, t.px1, t.py0, t.py1, r); ty = TileShape<3>::TY; break;
    default: interior_tiles<4>(nx, ny, t.px0, t.px1, t.py0, t.py1, r); ty = TileShape<4>::TY; break;
  }
  t.in_x0 = r[0];
  t.in_x1 = r[1];
  t.in_y0 = r[2];
  t.in_y1 = r[3];
  tiles.clear();
  for (int y = 0; y < (ny + ty - 1) / ty; ++y)
    for (int x = 0; x < (nx + 31) / 32; ++x)
      if (!(x >= r[0] && x < r[1] && y >= r[2] && y < r[3])) tiles.push_back(make_int2(x, y));
  t.n_edge = (int)tiles.size();
}

}  // namespace sllbm
