// Two 16-bit indices in one 32-bit word (host and device).
#pragma once

#if defined(__CUDACC__)
#define PM_HD __host__ __device__ __forceinline__
#else
#define PM_HD inline
#endif

// Cell (x, y) of a mesh of up to 46340 cells a side (n^2 < 2^31: a batch's
// instances; single meshes have up to 32768). The word is unsigned: rows from
// 32768 on reach its top bit.
PM_HD unsigned pack_cell(int x, int y) { return (unsigned)x | ((unsigned)y << 16); }
PM_HD int cell_x(unsigned w) { return (int)(w & 0xffffu); }
PM_HD int cell_y(unsigned w) { return (int)(w >> 16); }

// Offset (x, y) in cells, -32768 .. 32767.
PM_HD unsigned pack_offset(int x, int y) { return ((unsigned)x & 0xffffu) | ((unsigned)y << 16); }
PM_HD int offset_x(unsigned w) { return (int)(short)(w & 0xffffu); }
PM_HD int offset_y(unsigned w) { return (int)(short)(w >> 16); }
