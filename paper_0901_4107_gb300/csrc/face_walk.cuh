// The walk round a face of a convex cell held as triples of planes (dual triangles).
#pragma once

namespace amm {
namespace vor {

// Round plane k from vertex t0, a vertex's planes in tri (a | b << 8 | c << 16, in the
// order of the outward orientation): the vertex (k, x, y) is followed by (k, y, .), which
// next[k][y] names.  The table is not cleared between cells: an entry counts only if it
// is a vertex of this cell (live) with those planes.  visit(t) for each vertex after t0.
// Returns the number of vertices met, -1 for a walk that does not come back within `most`.
template <int P, typename Live, typename Visit>
__host__ __device__ __forceinline__ int walk_face(int k, int t0, const unsigned* tri, const unsigned char (*next)[P],
                                                  int most, Live live, Visit visit) {
  int t = t0, m = 0;
  for (;;) {
    const unsigned tr = tri[t];
    const int p0 = tr & 255, p1 = (tr >> 8) & 255, p2 = (tr >> 16) & 255;
    const int y = p0 == k ? p2 : (p1 == k ? p0 : p1);
    m++;
    const int tn = next[k][y];
    if (tn == t0) return m;
    if (m >= most || !live(tn)) return -1;
    const unsigned tq = tri[tn];
    const int g0 = tq & 255, g1 = (tq >> 8) & 255, g2 = (tq >> 16) & 255;
    if (!((g0 == k && g1 == y) || (g1 == k && g2 == y) || (g2 == k && g0 == y))) return -1;
    visit(tn);
    t = tn;
  }
}

// Did the walks of all planes, `walked` vertices together, meet every vertex on each of
// its three planes?  A walk that comes back meets each vertex of its plane at most once;
// a plane with vertices left over has a second cycle, and its face was not all of it.
__host__ __device__ __forceinline__ bool walks_complete(int walked, int vertices) { return walked == 3 * vertices; }

}  // namespace vor
}  // namespace amm
