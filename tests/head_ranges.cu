// Host side of the head ranges of the host-tensor step, run without a GPU: the descriptors are carved at an address that nothing reads, and
// what the launches would be given is looked at instead of launched.
#include <cuda_runtime.h>

#include <cstdio>
#include <type_traits>

template <class... A>
cudaError_t seen_launch(const cudaLaunchConfig_t* cfg, void (*kernel)(A...), A... args);
#define cudaLaunchKernelEx seen_launch
#define cudaGetLastError() cudaSuccess
#include "../paper_2602_01801_b200/csrc/update_kernels.cu"
#include "../paper_2602_01801_b200/csrc/fastar_api.cu"

static int bad = 0;
static const char* what = "";
static void expect(bool ok, const char* text) {
  if (!ok && bad++ < 20) std::printf("%s: %s\n", what, text);
}
static bool aligned(const void* p) { return !(reinterpret_cast<uintptr_t>(p) & 15); }

static UpdateScratch cleared;
template <class T>
void look(const T& v) {
  if constexpr (std::is_pointer_v<T>)
    if constexpr (std::is_object_v<std::remove_pointer_t<T>>)
      expect(sizeof(std::remove_pointer_t<T>) < 16 || aligned(v), "a launch gets a misaligned pointer to 16-byte pieces");
  if constexpr (std::is_same_v<T, UpdateScratch>) cleared = v;
}
template <class... A>
cudaError_t seen_launch(const cudaLaunchConfig_t*, void (*)(A...), A... args) {
  (look(args), ...);
  return cudaSuccess;
}
static CUresult no_map(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void* p, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                       CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return aligned(p) ? CUDA_SUCCESS : CUDA_ERROR_INVALID_VALUE;
}

int main() {
  int ranges = 0;
  for (int heads : {2, 3, 5, 11, 12, 20, 40})
    for (int max_tokens : {1, 77, 3111, 4200, 4725, 8201, 16383})
      for (int capacity : {16384, 128 * 513})
        for (int dtype : {FASTAR_BF16, FASTAR_FP32})
          for (int option = 0; option < 3; ++option) {
            fastar_cache c{};
            c.encode = no_map;
            c.desc = fastar_cache_desc{heads, option == 2 ? 64 : 128, capacity, option == 2 ? 64 : 128, 0, 4, option == 1 ? 8 : 5, max_tokens, 77, 3, dtype, 0,
                                       option == 1 ? 8 : 16, 0, option == 2 ? 1 : 0, 0};
            char name[160];
            std::snprintf(name, sizeof name, "%d heads, %d tokens, capacity %d, dtype %d, option %d", heads, max_tokens, capacity, dtype, option);
            what = name;
            expect(desc_valid(&c.desc), "descriptor");
            carve(c.desc, reinterpret_cast<uint8_t*>(1ull << 40), &c.v);
            for (int slices = 1; slices <= kMaxSlices && slices <= heads; ++slices)
              for (int i = 0; i < slices; ++i) {
                const int h0 = heads * i / slices, count = heads * (i + 1) / slices - h0;
                HeadRange r;
                expect(make_range(&c, h0, count, &r) == FASTAR_OK, "a tensor map would be refused");
                const CacheView& v = r.v;
                for (const void* p : {static_cast<void*>(v.cnt), static_cast<void*>(v.stamp), static_cast<void*>(v.count), static_cast<void*>(v.log2m),
                                      static_cast<void*>(v.rnorm), static_cast<void*>(v.hk), static_cast<void*>(v.hk_hi), static_cast<void*>(v.hq),
                                      static_cast<void*>(v.k8_new), static_cast<void*>(v.q8_ca), static_cast<void*>(v.q8_probe),
                                      static_cast<void*>(v.kp8_ca), static_cast<void*>(v.stage_prep)})
                  expect(aligned(p), "an array that is accessed in 16-byte pieces is misaligned");
                for (const __nv_bfloat16* p : v.stage) expect(aligned(p), "a staging slot is misaligned");
                expect((v.CAPB & 3) || (aligned(v.scores) && aligned(v.scores_hi)), "scores are misaligned");
                for (int n : {1, max_tokens}) {
                  cleared = UpdateScratch{};
                  expect(launch_prep_update(v, v.stage[0], n, static_cast<int64_t>(n) * v.D, v.D, nullptr) == 1, "launch");
                  const int64_t mt = max_tokens, cap = capacity;
                  expect(cleared.best == c.v.best + h0 * mt && cleared.n_best == count * mt, "not the range's own best matches are cleared");
                  if (!plan_is_fused(v, n)) {
                    expect(reinterpret_cast<int32_t*>(cleared.cnt) == c.v.cnt + h0 * cap && cleared.n_cnt16 == count * cap / 4, "not the range's own counters are cleared");
                    expect(cleared.n_match == c.v.n_match + h0 && cleared.n_heads == count, "not the range's own numbers of matches are cleared");
                  } else {
                    expect(cleared.n_cnt16 == 0 && cleared.n_heads == 0, "something is cleared that is not used");
                  }
                  ++ranges;
                }
              }
          }
  std::printf("%d ranges, %d findings\n", ranges, bad);
  return bad ? 1 : 0;
}
