// Columns of a strip of the strip-and-band sweep (included by demons_wide.cuh, inside its namespace).  Plain
// integer functions without CUDA headers, so that a host compiler can check them for every width.
#ifdef __CUDACC__
#define HR_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define HR_HOST_DEVICE inline
#endif

// First loaded column of the strip of output columns [x0, x1) at a level w pixels wide.  At the right edge the
// strip is shifted so that the three columns past the edge lie in the edge column's warp: an edge column in lane
// 29 .. 31 moves to lane 0 of the next one.
HR_HOST_DEVICE int strip_origin(int x0, int x1, int w)
{
    int xl = x0 - 6;   // u is exact from 3 columns inside, du's x pass from 6
    if (x1 == w) {
        const int past = ((w - 1 - xl) & 31) - 28;
        if (past > 0) xl -= 4 - past;
    }
    return xl;
}

// The column of the rows that thread t stands for: its own inside the image, the edge column outside, so that the
// three columns past an edge form the edge column's u and du.  X-pass rows are handed from lane to lane of a warp
// without a barrier, so a thread farther past the edge, whose values reach no output, keeps its own column
// where the edge column belongs to another warp.
HR_HOST_DEVICE int edge_column(int xl, int t, int w)
{
    const int x = xl + t, c = (x < 0 ? 0 : x > w - 1 ? w - 1 : x) - xl;
    return (c ^ t) < 32 ? c : t;
}
