// The allocation-free links on a scratch array with stale bin counts, as a call
// stopped between its kernels leaves them: the next call's links are those of a
// clean array.  argv[1]: file of int64 n, int64 n_rows, tpc_options, row radii, y,
// z (float), row, sector (uint8).  Prints "links <n> changed <n>".
#include <cstdio>
#include <vector>

#include "tpc_noalloc.cu"

template <typename T>
static std::vector<T> take(FILE* f, size_t n) {
  std::vector<T> v(n);
  if (fread(v.data(), sizeof(T), n, f) != n) {
    std::printf("short file\n");
    std::exit(1);
  }
  return v;
}

template <typename T>
static T* to_device(const std::vector<T>& v) {
  T* p = nullptr;
  if (cudaMalloc(&p, v.size() * sizeof(T)) != cudaSuccess ||
      cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess) {
    std::printf("no device memory\n");
    std::exit(1);
  }
  return p;
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
  std::vector<int32_t> got[2][2];
  for (int i = 0; i < 2; ++i) {
    int32_t* link[2];
    for (auto& l : link) l = to_device(std::vector<int32_t>(n, -7));
    if (tpc_links_noalloc(&geo, &opt, &cl, link[0], link[1], nullptr) != TPC_OK) return 1;
    for (int k = 0; k < 2; ++k) {
      got[i][k].resize(n);
      if (cudaMemcpy(got[i][k].data(), link[k], 4 * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    }
    // stale counts in every bin
    void* base = nullptr;
    if (scratch_address(&base) != cudaSuccess ||
        cudaMemset((char*)base + kOffBinCnt, 1, sizeof(int) * (kNoAllocBins + 1)) != cudaSuccess ||
        cudaDeviceSynchronize() != cudaSuccess)
      return 1;
  }
  long links = 0, changed = 0;
  for (size_t j = 0; j < n; ++j)
    for (int k = 0; k < 2; ++k) {
      links += got[0][k][j] >= 0;
      changed += got[0][k][j] != got[1][k][j];
    }
  std::printf("links %ld changed %ld\n", links, changed);
  return 0;
}
