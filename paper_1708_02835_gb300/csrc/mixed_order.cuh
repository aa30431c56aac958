// Which output tiles each update launch of one step of the mixed factorisation writes
// (factor_mixed in mixed.cu).  Also compiled for the host, where the two streams' order is
// checked tile by tile.
//
// Step k's updates C_mn -= P_m P_n^T fall into three parts:
//   kBandBand  both operands FP64 band tiles (m - k < band), on the side stream;
//   kColumn    column k + 1, and the corner: row m = k + band, columns k + 2 .. k + band;
//   kRest      everything else.
// kColumn and kRest run on the main stream, with the event that the next step's chain waits for
// between them.  The corner has to be ahead of that event: the chain of step k + 1 writes rows
// up to k + band in its own band x band update, and factors tile (k + 2, k + 2) after it, which
// for a band of two tiles is the corner.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define EGS_ORDER __host__ __device__ __forceinline__
#else
#define EGS_ORDER inline
#endif

namespace egs {
namespace order {

enum Part { kBandBand = 0, kColumn = 1, kRest = 2 };

// Columns of the corner of step k (0 if its row does not exist).
EGS_ORDER int corner_tiles(int k, int band, int T) { return k + band < T ? band - 1 : 0; }

// The FP64-accurate outputs of step k, enumerated: kBandBand, or those within xband >= band of
// the diagonal whose operands are not both FP64 band tiles.
EGS_ORDER int64_t band_tiles_of(int part, int k, int band, int xband, int T)
{
    if (part == kBandBand) {
        const int64_t nb = band - 1 < T - k - 1 ? band - 1 : T - k - 1;
        return nb * nb;
    }
    return part == kColumn ? xband + corner_tiles(k, band, T) : (int64_t)(T - k - 2) * xband;
}

// Tile t of them; false: not one of this part.
EGS_ORDER bool band_tile(int part, int k, int band, int xband, int T, int64_t t, int &m, int &n)
{
    if (part == kColumn && t >= xband) {
        m = k + band;
        n = k + 2 + (int)(t - xband);
        return true;
    }
    const int w = part == kBandBand ? (band - 1 < T - k - 1 ? band - 1 : T - k - 1) : xband;
    n = (part == kRest ? k + 2 : k + 1) + (int)(t / w);
    m = n + (int)(t % w);
    if (m >= T || (m - k < band) != (part == kBandBand)) return false;
    return !(part == kRest && m == k + band);
}

// Tiles enumerated by a launch of the tensor-core update (kColumn: column k + 1, then the corner,
// which with skip_band is another kernel's).
EGS_ORDER int64_t update_tiles_of(int part, int k, int band, int skip_band, int T)
{
    const int64_t r = T - k - 1;
    return part == kColumn ? r + (skip_band ? 0 : corner_tiles(k, band, T)) : (r - 1) * r / 2;
}

// Tile t >= T - k - 1 of kColumn: the corner.
EGS_ORDER void update_corner(int k, int band, int T, int64_t t, int &m, int &n)
{
    m = k + band;
    n = k + 2 + (int)(t - (T - k - 1));
}

// Whether an enumerated output (m, n) of the tensor-core update is one: neither band x band, nor
// (skip_band) within xband of the diagonal, nor in kRest the corner.
EGS_ORDER bool update_tile(int part, int k, int band, int m, int n, int skip_band, int xband)
{
    if (m - k < band) return false;
    if (skip_band && m - n < xband) return false;
    return !(part == kRest && m == k + band);
}

// With a band of one tile the diagonal tile k itself is an output of column k, so that its
// factorisation waits for the main stream; a wider band's diagonal tile is final once the
// chain's own band x band update and the corner before it are.
EGS_ORDER bool potrf_waits_for_column(int band) { return band == 1; }

}  // namespace order
}  // namespace egs
