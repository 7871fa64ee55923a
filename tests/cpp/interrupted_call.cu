// A tracking call that stops part-way (here at an event that does not exist, after
// the first launch), with bin counts and bids as its kernels would have left
// them in between: the next call gives a fresh context's tracks.  argv[1]: file
// of int64 n, int64 n_rows, tpc_options, row radii, y, z (float), row, sector (uint8).
// Prints "tracks <n> refs <n> changed <n>".
#include <cstdlib>

#include "tpc_api.cu"

template <typename T>
static std::vector<T> take(FILE* f, size_t n) {
  std::vector<T> v(n);
  if (fread(v.data(), sizeof(T), n, f) != n) std::exit(2);
  return v;
}

template <typename T>
static T* to_device(const std::vector<T>& v) {
  T* p = nullptr;
  if (cudaMalloc(&p, v.size() * sizeof(T)) != cudaSuccess ||
      cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess)
    std::exit(3);
  return p;
}

struct Result {
  std::vector<int> ids, attach;
  std::vector<float> par;
};

static Result track(tpc_ctx* ctx, const tpc_clusters& cl) {
  tpc_tracks out;
  if (tpc_track_timeframe(ctx, &cl, &out, nullptr, nullptr) != TPC_OK) std::exit(4);
  Result r;
  r.ids.resize(out.n_cluster_refs);
  r.attach.resize(cl.n);
  r.par.resize(5 * out.n_tracks);
  if (cudaMemcpy(r.ids.data(), out.cl_ids, 4 * r.ids.size(), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(r.attach.data(), out.attach, 4 * r.attach.size(), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(r.par.data(), out.params, 4 * r.par.size(), cudaMemcpyDeviceToHost) != cudaSuccess)
    std::exit(5);
  return r;
}

int main(int argc, char** argv) {
  FILE* f = argc > 1 ? fopen(argv[1], "rb") : nullptr;
  if (!f) return 1;
  const auto head = take<int64_t>(f, 2);
  const size_t n = (size_t)head[0];
  const tpc_options opt = take<tpc_options>(f, 1)[0];
  const auto rx = take<float>(f, (size_t)head[1]);
  const auto y = take<float>(f, n), z = take<float>(f, n);
  const auto row = take<uint8_t>(f, n), sec = take<uint8_t>(f, n);
  fclose(f);
  const tpc_geometry geo{36, (int32_t)rx.size(), rx.data()};
  const tpc_clusters cl{(int64_t)n, to_device(y), to_device(z), nullptr, to_device(row), to_device(sec)};
  tpc_ctx* ctx = nullptr;
  if (tpc_init(&geo, opt.bz, nullptr, &opt, &ctx) != TPC_OK) return 6;
  const Result want = track(ctx, cl);
  ctx->prof = true;  // (profiling without its events)
  tpc_tracks out;
  if (tpc_track_timeframe(ctx, &cl, &out, nullptr, nullptr) != TPC_ERR_CUDA) return 7;
  ctx->prof = false;
  if (cudaMemset(ctx->F.bin_cnt, 1, sizeof(int) * (ctx->F.cap_bins + 1)) != cudaSuccess ||
      cudaMemset(ctx->F.bid, 0, sizeof(unsigned long long) * ctx->cap_n) != cudaSuccess)
    return 8;
  const Result got = track(ctx, cl);
  const bool changed = got.ids != want.ids || got.attach != want.attach ||
                       got.par.size() != want.par.size() ||
                       std::memcmp(got.par.data(), want.par.data(), 4 * got.par.size()) != 0;
  std::printf("tracks %zu refs %zu changed %d\n", want.par.size() / 5, want.ids.size(), changed);
  tpc_destroy(ctx);
  return 0;
}
