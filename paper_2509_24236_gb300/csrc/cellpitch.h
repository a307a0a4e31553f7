// Row and plane pitch of the cell view's records.  Host code only, shared by
// the allocation and the launches, and compiled on its own by the host tests.
#pragma once

namespace pf {

struct CellPitch {
    int row;          // records from cell (i, j, k) to (i, j + 1, k)
    int plane;        // to (i, j, k + 1)
    long long count;  // records to allocate
};

// A warp-wide load of 32-byte records goes through L1 four lanes at a time,
// and the four lanes' records cost one pass for every distinct record in the
// same quarter of a 128-byte line (measured on L1-resident buffers: 8 cycles
// per warp-load when each group of four lanes reads one record or four in
// different quarters, 16 when it reads two in the same quarter, 32 when it
// reads four there).  Neighbouring points and particles fall in cells that
// are neighbours along any axis; with the node grid's pitch (nx a multiple of
// 4) two cells that differ along y or z always meet in one quarter.  So the
// row pitch is 2 and the plane pitch 3 modulo 4: the six neighbours of a cell
// and most diagonal ones fall in other quarters (simulated over multiroom
// frames, the passes per warp-load drop from 16.1 to 11.9 with lanes on
// points and from 10.1 to 8.1 with lanes on particles; with 16-byte records,
// which go eight lanes at a time, from 12.6 to 7.0 and from 5.4 to 4.1).
// Measured on multiroom, 3072 poses x 307 200 points: 2.95 -> 2.60 ms with
// lanes on points (28 -> 23 L1 wavefronts per warp-load, the rest being misses,
// the broadcast particles and shuffles), 1.67 -> 1.64 ms with lanes on
// particles; with a half-precision view of 317x233 points 242 -> 227 us.
// A cell's lower corner is never in the last column, row or plane of nodes,
// so nx - 1 records a row suffice and the pitched view of a grid of equal
// sides fits in the nx * ny * nz records an unpitched one has.  A grid whose
// pitched view would pass 2^31 records keeps the node grid's pitch (record
// indices are 32-bit), and so does one whose pitched view would need over a
// sixteenth more records than it has nodes: grids four to a dozen nodes wide,
// whose rows would grow by up to half.
inline CellPitch node_pitch(int nx, int ny, int nz) { return {nx, nx * ny, (long long)nx * ny * nz}; }

inline CellPitch cell_pitch(int nx, int ny, int nz)
{
    const long long nodes = (long long)nx * ny * nz;
    const long long row = (nx - 1) + ((2 - (nx - 1)) & 3);
    const long long rows = row * (ny - 1);
    const long long plane = rows + ((3 - rows) & 3);
    const long long last = (long long)(nx - 2) + row * (ny - 2) + plane * (nz - 2);
    if (last + 1 >= 2147483648LL || last + 1 > nodes + nodes / 16) return node_pitch(nx, ny, nz);
    return {(int)row, (int)plane, last + 1 > nodes ? last + 1 : nodes};
}

// The cell view of a volume: 1 the full view, 2 the narrow one, -1 none.
struct CellView {
    int mode;
    CellPitch pitch;
};

// Automatic choice within `budget` bytes, for a grid and weights of grid_bytes
// and records of narrow_bytes, with wide_bytes more each in the full view (0:
// the two views are the same): the full view when it fits, else the narrow one,
// else none.  The node pitch stands in where the pitched view misses the budget
// and it does not, so the pitch decides no view away.
inline CellView choose_view(int nx, int ny, int nz, long long grid_bytes, long long narrow_bytes, long long wide_bytes,
                            long long budget)
{
    const CellPitch pitches[2] = {cell_pitch(nx, ny, nz), node_pitch(nx, ny, nz)};
    for (int mode = 1; mode <= (wide_bytes ? 2 : 1); ++mode)
        for (const CellPitch& p : pitches)
            if (grid_bytes + p.count * (narrow_bytes + (mode == 1 ? wide_bytes : 0)) <= budget) return {mode, p};
    return {-1, pitches[0]};
}

}  // namespace pf
