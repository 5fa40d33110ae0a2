// Host-side table builders (double precision, no fused multiply-adds).
#pragma once

#include <stdint.h>

#include <vector>

#include "bf_internal.h"

namespace bfi {

struct GeomHost {
    int ne = 0;
    std::vector<double> xe;  // element x positions (m)
    double fnum = 1.0;
    int nx = 1, nz = 1;
    double x0 = 0, x1 = 0, z0 = 0, z1 = 0;
    double fs = 0, f0 = 0, c = 0;
};

// Angle-independent tables of a handle.
struct GeometryHost {
    std::vector<int> ap_first;     // [nx][ne] first row inside the aperture (nz: never)
    std::vector<uint16_t> apcnt;   // [nx][nz] channels inside the aperture
    std::vector<float> rowZ;
    std::vector<float> dx2;        // [ne][nxp] (kappa (x_p - x_i))^2, columns padded
};

// Tables of one angle set and sample count.  Row: the type rows are stored in.
template <class Row>
struct PlanHost {
    std::vector<int> colK, rowK;
    std::vector<float> colF, rowF;
    std::vector<Row> valid;        // [na][ne][nxp][2] first / last counted row (padding: none)
    int nsp = 0;
};

// Envelope transform of a depth: length 2^lg and the spectral factors of
// EnvJob (gr only with a band).
struct EnvHost {
    int lg = 0, conv = 0;
    std::vector<float> gr, gh;
};

double grid_coord(double lo, double hi, int n, int j);
void geometry_tables(const GeomHost &g, GeometryHost &out);
// Window of sample pairs a tile of tile_rows rows needs per run of `run` adjacent
// channels, and the width of the tensor copies it is fetched in.
void tile_window(const GeomHost &g, const std::vector<double> &angles, int prec, int tile_rows,
                 int run, int &wmax, int &box);
// (Row: int16_t for the device, whose grids are below 2^15 rows, or int)
template <class Row>
void angle_tables(const GeomHost &g, const GeometryHost &geo, int ns,
                  const std::vector<double> &angles, PlanHost<Row> &out);
// Channels per pipeline stage whose sample windows take stage_bytes.
int stage_channels(int wmax, int prec, int rows_per_thread, int stage_bytes, int ne);
void bandpass_bins(int nz, double z0, double z1, double c, double f0, int &lo, int &hi);
// Plane-wave f-k mapping of every (angle, Kz bin q = 1 .. nt/2, Kx bin m):
// i0 [na][nt/2][nk] the temporal bin below the mapped position (-1: nothing
// taken), aw [na][nt/2][nk][2] its interpolation weight toward i0 + 1 and the
// spectral weight.  sc: sin, cos of each angle.  stolt: Stolt's mapping of the
// exploding-reflector fit instead of the exact plane-wave mapping.  Double
// precision, evaluated in the order the definitions are written.  lgk > 0: transposed,
// [na][nk][nt/2], Kx bins in the order of fk_kx_bin.
void fk_mapping_tables(int nt, int nk, double pitch, double dz, const std::vector<double> &sc,
                       bool stolt, int lgk, std::vector<int> &i0, std::vector<float> &aw);
// exp(-2 pi i k / n) for k < n, interleaved.
void fft_twiddles(int n, std::vector<float> &tw);
// The level twiddles of every Fft16 transform (layout: bf_fft16.cuh), interleaved.
void fft16_twiddles(std::vector<float> &tw);
// band: keep the bins lo .. hi only.
void envelope_tables(int nz, bool band, int lo, int hi, EnvHost &out);

}  // namespace bfi
