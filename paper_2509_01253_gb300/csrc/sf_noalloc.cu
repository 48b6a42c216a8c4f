// sf_noalloc.cu -- rotation (automorphism + key switching) that allocates no
// device memory.
//
// Some callers cannot call cudaMalloc: code running inside a stream-ordered
// allocator's or a host framework's memory budget that must not grow, plug-ins
// loaded into a process whose allocator owns the whole device, and real-time
// paths where an allocation (or the synchronising cudaFree that a growing
// workspace implies) would stall.  sf_rotate_noalloc serves them: its scratch
// is the fixed array below, reserved once per GPU when the library's module
// is loaded on that GPU, and every call reuses it.
#include <algorithm>
#include <mutex>

#include "sf_internal.h"
#include "sf_ks.h"

// 32 MiB of scratch per GPU that loads this library, held until the process exits.
#define SF_NOALLOC_SCRATCH_WORDS ((size_t)4 << 20)
static __device__ __align__(256) u64 g_sf_noalloc_scratch[SF_NOALLOC_SCRATCH_WORDS];

#define SF_NOALLOC_MAX_DEVICES 64
static u64 *g_noalloc_ptr[SF_NOALLOC_MAX_DEVICES];
static std::mutex g_noalloc_mu;

// Device address of the array on `device` (which must be current).  In host
// code the array's name is only a host-side stand-in, so the address has to
// come from cudaGetSymbolAddress, once per device.
static sf_status noalloc_scratch(int device, u64 **out)
{
    if (device < 0 || device >= SF_NOALLOC_MAX_DEVICES) return sf_set_error(SF_EINVAL, "device %d out of range", device);
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[device]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_sf_noalloc_scratch);
        if (e != cudaSuccess || !p)
            return sf_set_error(SF_ECUDA, "cudaGetSymbolAddress of the no-alloc scratch failed: %s", cudaGetErrorString(e));
        g_noalloc_ptr[device] = (u64 *)p;
    }
    *out = g_noalloc_ptr[device];
    return SF_OK;
}

static inline size_t round_words(size_t w) { return (w + 31) & ~(size_t)31; }

extern "C" sf_status sf_rotate_noalloc(sf_ctx *ctx, const sf_rotkeys *rk, int32_t d, const uint64_t *d_ct,
                                       uint64_t *d_out, int32_t count, void *stream)
{
    if (!ctx) return sf_set_error(SF_EINVAL, "sf_rotate_noalloc: null context");
    SF_CUDA_TRY(cudaSetDevice(ctx->device));
    const SfRing &R = ctx->ring;
    if (!rk || rk->ctx != ctx || !d_ct || !d_out || count < 1) return sf_set_error(SF_EINVAL, "sf_rotate_noalloc: bad arguments");
    int slot = -1;
    for (size_t t = 0; t < rk->d.size(); ++t)
        if (rk->d[t] == d) slot = (int)t;
    if (slot < 0) return sf_set_error(SF_EINVAL, "no rotation key for d = %d", d);
    const size_t ct = (size_t)2 * R.L * R.n;
    // key switches run in launch batches of the context's size, as in sf_rotate
    const int batch = std::min(ctx->ks_batch, (int)count);
    // what the call uses: the workspaces of one launch batch, then room for a copy of
    // the input (buffers that share words)
    const size_t ks_words = round_words(sf_ks_scratch_words(R) * batch), used = ks_words + round_words((size_t)count * ct);
    // the documented limit, which stays as it is: two ciphertexts and this many
    // key-switch limbs per call
    const size_t limbs = R.L + std::max(R.L, 2 * R.K) + std::max(R.dnum * R.nm, 2 * R.L) + 2 * R.L;
    const size_t limit = 2 * round_words((size_t)count * ct) + round_words((limbs << R.log_n) * batch);
    if (std::max(used, limit) > SF_NOALLOC_SCRATCH_WORDS)
        return sf_set_error(SF_EINVAL,
                            "sf_rotate_noalloc: %d ciphertexts are beyond the documented limit: two ciphertexts each and their "
                            "key-switch workspaces are %zu bytes, the fixed maximum is %zu bytes",
                            count, std::max(used, limit) * sizeof(u64), SF_NOALLOC_SCRATCH_WORDS * sizeof(u64));
    u64 *ws = nullptr;
    SF_TRY(noalloc_scratch(ctx->device, &ws));
    cudaStream_t st = (cudaStream_t)stream;
    // per-launch event bracketing would create CUDA events; keep this call free of that
    const int timing = ctx->kernel_timing;
    ctx->kernel_timing = 0;
    sf_status s = SF_OK;
    const bool copy = sf_words_overlap(d_ct, d_out, ct * count);
    u64 *in = ws + ks_words;
    if (copy && cudaMemcpyAsync(in, d_ct, sizeof(u64) * ct * count, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        s = sf_set_error(SF_ECUDA, "sf_rotate_noalloc: copying the input failed: %s", cudaGetErrorString(cudaGetLastError()));
    if (s == SF_OK) {
        SfKsBatch b;
        memset(&b, 0, sizeof(b));
        b.E = copy ? in : d_ct;
        b.E_stride = ct;
        b.out = d_out;
        b.out_stride = ct;
        b.inner = 1 << 30;
        b.count = count;
        b.d = d;
        b.add_v = 0;
        b.unreduced = 1;   // no sf_check_residues here
        b.key = rk->d_keys + rk->key_words * slot;
        s = sf_ks_run(ctx, b, ws, batch, st);
    }
    ctx->kernel_timing = timing;
    return s;
}
