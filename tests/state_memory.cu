// Batches on a device with little memory left, checked through the library's own
// objects linked with a cudaMalloc that refuses what a limit forbids (the
// failure is made on the host: the device's memory stays free).  A batch whose
// state buffer cannot be had runs in another shape, with the same results, and
// what the context already holds stays where it is, call after call.
// Prints one line per check that fails; exits 0 if there is none.
#include <cstdio>
#include <cstring>
#include <vector>

#include "fire_internal.h"

static size_t g_limit = ~(size_t)0;   // largest allocation granted

extern "C" cudaError_t __real_cudaMalloc(void **p, size_t n);
extern "C" cudaError_t __wrap_cudaMalloc(void **p, size_t n)
{
    if (n > g_limit) {
        *p = nullptr;
        return cudaErrorMemoryAllocation;
    }
    return __real_cudaMalloc(p, n);
}

static int g_failed = 0;
static void check(bool ok, const char *what, int size)
{
    if (!ok) {
        g_failed = 1;
        printf("%d x %d: %s\n", size, size, what);
    }
}

int main()
{
    const int n = 2000;
    // 256 tiles: the state also fits in shared memory; 1024: it does not
    for (int size : {512, 1024}) {
        const size_t hw = (size_t)size * size;
        std::vector<uint8_t> veg(hw, 2);
        std::vector<float> zero(hw, 0.0f);
        fire_ctx *ctx = nullptr;
        fire_map *map = nullptr;
        if (fire_create(&ctx, 0, nullptr) ||
            fire_maps_upload(ctx, size, size, 30.0f, veg.data(), zero.data(), zero.data(),
                             zero.data(), zero.data(), 0, &map)) {
            printf("set-up: %s\n", fire_last_error(ctx));
            return 1;
        }
        std::vector<fire_params> p(n, fire_params{{-1.2, 0.0, 0.0, 0.5, 0.0}});
        std::vector<fire_cell> c(n, fire_cell{size / 2, size / 3});
        std::vector<uint64_t> s(n);
        for (int i = 0; i < n; ++i) s[i] = 100 + i;
        fire_params *dp;
        fire_cell *dc;
        uint64_t *ds;
        fire_result *out;
        if (cudaMalloc((void **)&dp, n * sizeof *dp) || cudaMalloc((void **)&dc, n * sizeof *dc) ||
            cudaMalloc((void **)&ds, n * sizeof *ds) || cudaMalloc((void **)&out, n * sizeof *out))
            return 1;
        cudaMemcpy(dp, p.data(), n * sizeof *dp, cudaMemcpyHostToDevice);
        cudaMemcpy(dc, c.data(), n * sizeof *dc, cudaMemcpyHostToDevice);
        cudaMemcpy(ds, s.data(), n * sizeof *ds, cudaMemcpyHostToDevice);
        std::vector<fire_result> want(n), got(n);
        auto run = [&](fire_ctx *x, std::vector<fire_result> &r) {
            cudaMemset(out, 0xff, n * sizeof *out);
            const int rc = fire_simulate_batch(x, map, n, dp, dc, ds, 0,
                                               FIRE_DEVICE_PTRS | FIRE_SYNC, out, nullptr);
            cudaMemcpy(r.data(), out, n * sizeof *out, cudaMemcpyDeviceToHost);
            return rc;
        };
        check(run(ctx, want) == FIRE_OK, "reference call", size);
        check(want[0].burnt > 1 && cudaGetLastError() == cudaSuccess, "reference fires", size);

        // a second context, which holds a state buffer for a few fires first
        fire_ctx *low = nullptr;
        if (fire_create(&low, 0, nullptr)) return 1;
        const size_t per_block = (size_t)map->dev.ntiles * 256;
        fire_set_launch(low, 4, 1, 0, FIRE_STATE_GLOBAL);
        check(fire_simulate_batch(low, map, 8, dp, dc, ds, 0, FIRE_DEVICE_PTRS | FIRE_SYNC,
                                  out, nullptr) == FIRE_OK, "first call", size);
        fire_set_launch(low, 0, 0, 0, FIRE_STATE_AUTO);
        g_limit = 20 * per_block;
        for (int call = 0; call < 2; ++call) {
            check(run(low, got) == FIRE_OK, "call with little memory", size);
            check(!memcmp(want.data(), got.data(), n * sizeof want[0]), "results", size);
        }
        const uint32_t *held = low->gstate;
        const unsigned long long epoch = (unsigned long long)low->epoch;
        check(run(low, got) == FIRE_OK && low->gstate == held &&
                  (unsigned long long)low->epoch == epoch,
              "buffer kept from call to call", size);
        check(low->gstate_bytes <= 20 * per_block, "buffer within the limit", size);
        // memory comes back: the full shape again
        g_limit = ~(size_t)0;
        check(run(low, got) == FIRE_OK && low->gstate_bytes > 100 * per_block,
              "full shape with memory back", size);
        check(!memcmp(want.data(), got.data(), n * sizeof want[0]), "results", size);
        // nothing at all: an error, and the context usable
        fire_ctx *none = nullptr;
        if (fire_create(&none, 0, nullptr)) return 1;
        g_limit = 4096;
        const int rc = run(none, got);
        check(size == 512 ? rc == FIRE_OK : rc == FIRE_ENOMEM, "no memory", size);
        g_limit = ~(size_t)0;
        check(run(none, got) == FIRE_OK, "after it", size);
        check(!memcmp(want.data(), got.data(), n * sizeof want[0]), "results", size);
        fire_destroy(none);
        fire_destroy(low);
        fire_map_free(map);
        fire_destroy(ctx);
        cudaFree(dp);
        cudaFree(dc);
        cudaFree(ds);
        cudaFree(out);
    }
    return g_failed;
}
