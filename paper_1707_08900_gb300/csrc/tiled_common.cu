// Tile tables of the tiled substep kernels and TMA descriptor encoding.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>

#include "tiled.cuh"

namespace gbfd {

namespace {

// (tx, ty, ns) variants compiled per storage width; each is offered with
// several z-chunk lengths.
const TileConfig kVariants4[] = {{32, 8, 0, 9, 1},
                                 {32, 8, 0, 8, 2, 2},
                                 {32, 8, 0, 8, 2, 2, 0, 1},
                                 {32, 8, 0, 8, 2, 1, 0, 1},
                                 {32, 8, 0, 8, 2, 2, 1, 1},
                                 {32, 8, 0, 8, 2, 2, 1, 1},
                                 {32, 8, 0, 8, 2, 2, 1, 1}};
const TileConfig kVariants8[] = {{32, 4, 0, 8, 1},       {16, 8, 0, 8, 1},
                                 {32, 4, 0, 6, 2, 1},    {32, 4, 0, 5, 2, 2},
                                 {32, 8, 0, 5, 2, 1},    {16, 8, 0, 5, 1, 0, 1, 1}};
const int kZc[kZcChoices] = {40, 32, 64, 16, 8};
constexpr int kNz = kZcChoices;

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

}  // namespace

int tiled_config_count(int sbytes)
{
    return (sbytes == 8 ? (int)(sizeof kVariants8 / sizeof kVariants8[0])
                        : (int)(sizeof kVariants4 / sizeof kVariants4[0])) *
           kNz;
}

TileConfig tiled_config(int sbytes, int i)
{
    TileConfig t = sbytes == 8 ? kVariants8[i / kNz] : kVariants4[i / kNz];
    t.zc = kZc[i % kNz];
    return t;
}

namespace {

// Time of a launch in plane times, from the list schedule of its CTAs: tiles
// columns of nz planes in chunks of zc, `per` CTAs per SM, a CTA costing its
// planes plus h (the six halo planes, which only load and add to the z-paired
// terms, and the start-up), the short last chunks last.  share[k]: the time of
// a CTA with k on its SM, in units of that with `per`.
double launch_time(long long tiles, int nz, int zc, int sms, int per, double h, double odd,
                   const double *share)
{
    const long long slots = (long long)sms * per;
    const long long chunks = (nz + zc - 1) / zc, whole = tiles * (chunks - 1);
    const int last = nz - zc * (int)(chunks - 1);
    const double c = zc + h + odd * (zc % 2), cl = last + h + odd * (last % 2);
    auto part = [&](long long r) { return share[std::min<long long>(per, (r + sms - 1) / sms)]; };
    const double t0 = (double)(whole / slots) * c;
    const long long r = whole % slots;  // whole chunks beside the first last chunks
    long long left = tiles;
    if (r == 0)
        return t0 + (double)(left / slots) * cl + (left % slots ? cl * part(left % slots) : 0.0);
    const long long idle = slots - r;
    if (left <= idle)
        return t0 + std::max(c, cl) * part(r + left);
    const int k = (int)(c / cl);  // last chunks an idle slot takes meanwhile
    left -= idle * k;
    if (left <= 0)
        return t0 + c;
    const double t = t0 + std::max(c, (k + 1) * cl);
    if (left <= idle)
        return t;
    if (left <= slots)
        return std::max(t, t0 + c + cl * part(left));
    return t + cl + (double)((left - slots) / slots) * cl;
}

}  // namespace

// Chosen by launch_time with the shares measured on small grids: two FP32 CTAs
// per SM (one alone runs at 0.8 of the time), three FP64 ones, whose SM's FP64
// pipe one CTA nearly fills.  Odd lengths cost the FP32 kernel half a plane
// (two planes per loop iteration).  Where lengths of 24 (FP32) or 10 (FP64)
// planes and more give 6 or 3 full waves, only those are looked at: with fewer
// waves of long columns the model misses how far apart in z the CTAs drift,
// and the halo rows they share leave L2.  Against the best of up to 36 lengths
// timed on 14 grids from 16^3 to 512^3 the choice is within 1.3% (FP32) and
// 1.9% (FP64) on the geometric mean, us per substep:
//   FP32  96^3 26.1 -> 21.3, 160^3 84.5 -> 72.8, 512^3 1944 -> 1907,
//         200 x 136 x 105 82.4 -> 75.8 (before: 64, 40, 32, 16 or 8 planes by
//         the number of waves);
//   FP64  16^3 185 -> 22.5, 32^3 360 -> 32.8, 64^3 447 -> 174, 128^3 1246 ->
//         1182 (before: 40 planes always).
int default_zc(int w, long long tiles, int nz, int sms)
{
    const double share32[3] = {0.0, 0.8, 1.0}, share64[4] = {0.0, 0.36, 0.75, 1.0};
    const bool f32 = w == 4;
    const int per = f32 ? 2 : 3, min_zc = f32 ? 24 : 10, waves = f32 ? 6 : 3;
    int best = nz;
    double best_t = 1e300;
    bool many = false;  // some length fills the waves: the others no longer count
    for (int zc = 1; zc <= nz && zc <= 160; ++zc) {
        if (f32 && zc % 2 && zc != 1 && zc != nz)
            continue;
        const bool full = zc >= min_zc &&
                          tiles * ((nz + zc - 1) / zc) >= (long long)waves * per * sms;
        if (many && !full)
            continue;
        const double t = launch_time(tiles, nz, zc, sms, per, f32 ? 3.0 : 0.4, f32 ? 0.5 : 0.0,
                                     f32 ? share32 : share64);
        // (longer chunks read fewer halo planes: they win ties)
        if (t <= best_t || (full && !many)) {
            best_t = t;
            best = zc;
        }
        many = many || full;
    }
    return best;
}

namespace {

bool encode_tmap(TmapCache *cache, const void *origin, const Layout &L, int nf, int bx, int by,
                 int key, CUtensorMap **out)
{
    for (int i = 0; i < TmapCache::kEntries; ++i) {
        TmapCache::Entry &e = cache->e[i];
        if (e.valid && e.base == origin && e.cfg == key && e.nf == nf) {
            *out = &e.map;
            return true;
        }
    }
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn)
        return false;
    TmapCache::Entry &e = cache->e[cache->next];
    cache->next = (cache->next + 1) % TmapCache::kEntries;
    memset(&e, 0, sizeof e);
    // with walls in z the map covers the ghost planes too: it starts at
    // ghost plane -gz (kernels add gz to the plane index)
    const cuuint64_t dims[4] = {(cuuint64_t)(L.nx + 2 * GX), (cuuint64_t)L.rows,
                                (cuuint64_t)(L.nz + 2 * L.gz), (cuuint64_t)nf};
    const char *base = static_cast<const char *>(origin) - (long long)L.gz * L.plane * L.w;
    const cuuint64_t strides[3] = {(cuuint64_t)(L.P * L.w), (cuuint64_t)(L.plane * L.w),
                                   (cuuint64_t)(L.fpitch * L.w)};
    const cuuint32_t box[4] = {(cuuint32_t)bx, (cuuint32_t)by, 1u, (cuuint32_t)nf};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = fn(&e.map, L.w == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                    4, const_cast<char *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        return false;
    e.base = origin;
    e.cfg = key;
    e.nf = nf;
    e.valid = true;
    *out = &e.map;
    return true;
}

}  // namespace

bool get_state_tmap(TmapCache *cache, const void *origin, const Layout &L, int nf, int tx, int ty,
                    int cfg_key, CUtensorMap **out)
{
    return encode_tmap(cache, origin, L, nf, tx + 2 * GX, ty + 2 * GY, cfg_key, out);
}

bool get_tile_tmap(TmapCache *cache, const void *origin, const Layout &L, int nf, int tx, int ty,
                   int cfg_key, CUtensorMap **out)
{
    return encode_tmap(cache, origin, L, nf, tx, ty, 1000 + cfg_key, out);
}

}  // namespace gbfd
