// k_double2d.cu -- two steps per pass for large 2-D ideal-MHD FP32 domains, single and
// batched (D2Q5), as k_ideal_double (k_ideal.cu) does in 3-D.
//
// One step reads and writes 40 populations a cell and runs at the copy rate of HBM; this
// pass reads and writes them once for an even and an odd step, from one buffer (parity 0)
// to the other (parity 0).  A warp walks up a strip of at most 30 cells on its own: row by
// row every lane (the strip and one cell on either side) loads its cell's populations and
// collides them (step 1); what step 1 sends along x reaches the neighbouring lanes by
// shuffles, what it sends along y and keeps at rest stays in the lane's registers; the row
// below then has all that step 1 sent to it, is collided again (step 2) and stored where
// the next even step reads it (slot i of x + c_i).  No barrier and no shared memory but
// for the domain's constants; strips of 30 x rows redo 2 cells a row and 2 rows a strip.
// The arithmetic is ideal_collide_f32's: the result is that of two single steps bit for
// bit.  Measured, two-step passes against single steps: 64 domains of 64^2 .. 1024^2, 64
// steps with fields in and out, 68.5 -> 42.9 ms; 1000^2, 64 steps 3.10 -> 2.08 ms; 2048^2
// 12.9 -> 9.0; 4096^2, 32 steps 26.9 -> 19.9.  Strips of 16 rows: of 8 as fast, of 32, 64
// and 128 at 2048^2 9.6, 12.0 and 16.6 ms (neighbouring strips drift apart, and their
// shared lines leave L2 in between).
#include <algorithm>

#include "ideal_cell.cuh"

namespace vlbm {
namespace {

constexpr int kStripX = 30;
constexpr int kStripRows = 16;
constexpr int kStripThreads = 128;  // four strips a CTA

struct StripDomain {
    int nx, ny, tile_x;
    int64_t offset, stride;
    float gm1;
    RelaxSource relax[8];
};

__global__ void __launch_bounds__(kStripThreads, 4) k_double_2d(const float *__restrict__ in, float *__restrict__ out,
                                                                const int4 *__restrict__ tiles, int ntiles,
                                                                const StripDomain *__restrict__ doms, unsigned *flags)
{
    constexpr int Q = 5;
    __shared__ RelaxSource constants[kStripThreads / 32][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = blockIdx.x * (kStripThreads / 32) + warp;
    if (t >= ntiles) return;
    const int4 tile = tiles[t];  // domain, first cell of the strip, first row
    const StripDomain *d = doms + tile.x;
    if (lane < 8) constants[warp][lane] = d->relax[lane];
    __syncwarp();
    auto relax = [&](int k) { return constants[warp][k]; };
    const int nx = d->nx, ny = d->ny, x0 = tile.y, y0 = tile.z;
    const int xe = min(x0 + d->tile_x, nx), ye = min(y0 + kStripRows, ny);
    const float gm1 = d->gm1;
    const int64_t stride = d->stride;
    in += d->offset;
    out += d->offset;
    int x = x0 - 1 + lane;
    const bool first = x <= xe, second = lane >= 1 && x < xe;
    x += x < 0 ? nx : (x >= nx ? -nx : 0);
    const uint32_t row = (uint32_t)nx;  // cells of a domain fit 32 bits
    const uint32_t xm = (uint32_t)(x > 0 ? x - 1 : nx - 1), xp = (uint32_t)(x + 1 < nx ? x + 1 : 0);
    // of the row below: at rest, sent along +x and -x to this cell; sent up from it and from the one below that
    float rest[8], fromm[8], fromp[8], up1[8], up2[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) rest[k] = fromm[k] = fromp[k] = up1[k] = up2[k] = 0.f;
    for (int y = y0 - 1; y <= ye; ++y) {
        float f[8][Q];
        if (first) {
            const float *p = in + ((uint32_t)x + row * (uint32_t)(y < 0 ? y + ny : (y >= ny ? y - ny : y)));
#pragma unroll
            for (int k = 0; k < 8; ++k)
#pragma unroll
                for (int i = 0; i < Q; ++i) f[k][i] = p[(int64_t)(k * Q + i) * stride];
            ideal_collide_f32<2>(f, gm1, relax, flags);
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k)
#pragma unroll
                for (int i = 0; i < Q; ++i) f[k][i] = 0.f;
        }
        // what step 2 of the row below gets; f[k][4] is already what this row sends down
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float r = f[k][0], u = f[k][3];
            const float m = __shfl_up_sync(0xffffffffu, f[k][1], 1), q = __shfl_down_sync(0xffffffffu, f[k][2], 1);
            f[k][0] = rest[k];
            f[k][1] = fromm[k];
            f[k][2] = fromp[k];
            f[k][3] = up2[k];
            rest[k] = r;
            fromm[k] = m;
            fromp[k] = q;
            up2[k] = up1[k];
            up1[k] = u;
        }
        if (y > y0 && second) {
            ideal_collide_f32<2>(f, gm1, relax, flags);
            const uint32_t yo = (uint32_t)(y - 1), at = row * yo;
            const uint32_t up = row * (yo + 1 < (uint32_t)ny ? yo + 1 : 0u), dn = row * (yo > 0 ? yo - 1 : (uint32_t)ny - 1);
            const uint32_t to[Q] = {(uint32_t)x + at, xp + at, xm + at, (uint32_t)x + up, (uint32_t)x + dn};
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                float *o = out + to[i];
#pragma unroll
                for (int k = 0; k < 8; ++k) o[(int64_t)(k * Q + i) * stride] = f[k][i];
            }
        }
    }
}

int strip_width(int nx)
{
    const int n = (nx + kStripX - 1) / kStripX;
    return (nx + n - 1) / n;
}

}  // namespace

// Where the pass is taken: 2-D FP32 domains that together exceed L2, with strips that fill
// the device: of the cells that all waves of warps could produce, rims and end rows
// included, at least 0.6 are wanted cells.  The gain is proportional to that share: 1.60 for
// the 64 domains above (0.79), 1.44 at 1000^2 (0.76).  Eleven other domains, 920^2 .. 4096^2, thin ones
// among them: 1.34 .. 1.48; six batches of equal domains 64^2 .. 600^2: 1.48 .. 1.58.
bool double_2d_ok(vlbm_ctx *c)
{
    if (c->model != VLBM_IDEAL || c->nlat != 8 || c->dim != 2 || c->storage != VLBM_F32 || c->slab || c->closure ||
        c->solid || any_open_face(c) || c->pop_bytes < (size_t(128) << 20))
        return false;
    if (c->double_slots == 0) {
        c->double_slots = -1;
        int dev = 0, sms = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_double_2d, kStripThreads, 0) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        const int64_t slots = (int64_t)sms * per_sm * (kStripThreads / 32);
        int64_t strips = 0, cells = 0;
        bool fits = slots > 0;
        for (const Domain &d : c->dom) {
            const int w = strip_width(d.nx);
            strips += (int64_t)((d.nx + w - 1) / w) * ((d.ny + kStripRows - 1) / kStripRows);
            cells += d.ncell;
            fits = fits && d.ncell < (int64_t(1) << 31);
        }
        if (!fits || strips > (int64_t(1) << 28)) return false;
        const int64_t waves = (strips + slots - 1) / slots;
        if ((double)cells >= 0.6 * (double)waves * slots * kStripX * (kStripRows + 2)) c->double_slots = (int)slots;
    }
    return c->double_slots > 0;
}

// The strip table and the domains' constants on the device, when the context is created.
vlbm_status double_2d_prepare(vlbm_ctx *c)
{
    std::vector<StripDomain> doms;
    std::vector<int4> tiles;
    std::vector<int> order(c->dom.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return c->dom[a].ncell > c->dom[b].ncell; });
    for (const Domain &dm : c->dom) {
        StripDomain s{};
        s.nx = dm.nx;
        s.ny = dm.ny;
        s.tile_x = strip_width(dm.nx);
        s.offset = dm.offset;
        s.stride = dm.stride;
        s.gm1 = (float)(dm.gamma - 1.0);
        for (int k = 0; k < 8; ++k)
            s.relax[k] = relax_source<2>((float)(1.0 / dm.tau[k]), (float)(AxisSet<2>::w0 * dm.source[k]),
                                         (float)(AxisSet<2>::w1 * dm.source[k]));
        doms.push_back(s);
    }
    for (int i : order)  // large domains first, small ones fill the tail
        for (int y = 0; y < doms[i].ny; y += kStripRows)
            for (int x = 0; x < doms[i].nx; x += doms[i].tile_x) tiles.push_back(make_int4(i, x, y, 0));
    const size_t dom_bytes = doms.size() * sizeof(StripDomain), tile_at = (dom_bytes + 15) / 16 * 16;
    const size_t bytes = tile_at + tiles.size() * sizeof(int4);
    void *blk = nullptr;
    if (c->params.alloc) {
        blk = c->params.alloc(bytes, (void *)c->stream, c->params.alloc_user);
    } else if (cudaMalloc(&blk, bytes) != cudaSuccess) {
        cudaGetLastError();
        blk = nullptr;
    }
    if (!blk) return fail(c, VLBM_ERR_OOM, "strip table allocation failed");
    c->owned.emplace_back(blk, bytes);
    char *p = static_cast<char *>(blk);
    vlbm_status s = cuda_check(c, cudaMemcpyAsync(p, doms.data(), dom_bytes, cudaMemcpyHostToDevice, c->stream),
                               "strip domains upload");
    if (s == VLBM_OK)
        s = cuda_check(c, cudaMemcpyAsync(p + tile_at, tiles.data(), tiles.size() * sizeof(int4), cudaMemcpyHostToDevice,
                                          c->stream),
                       "strip table upload");
    if (s == VLBM_OK) s = cuda_check(c, cudaStreamSynchronize(c->stream), "strip table upload");
    if (s != VLBM_OK) return s;
    c->double_doms = p;
    c->double_tiles = p + tile_at;
    c->double_ntiles = (int)tiles.size();
    return VLBM_OK;
}

vlbm_status double_2d(vlbm_ctx *c, const void *in, void *out)
{
    constexpr int per = kStripThreads / 32;
    k_double_2d<<<(unsigned)((c->double_ntiles + per - 1) / per), kStripThreads, 0, c->stream>>>(
        static_cast<const float *>(in), static_cast<float *>(out), static_cast<const int4 *>(c->double_tiles),
        c->double_ntiles, static_cast<const StripDomain *>(c->double_doms), c->d_flags);
    c->launches++;
    return cuda_check(c, cudaGetLastError(), "2-D two-step launch");
}

}  // namespace vlbm
