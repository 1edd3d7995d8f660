// Device construction of the 27-entry neighbour table of the leaf Blocks
// (Sec. II.B: each Block's ghost data comes from neighbouring Blocks of the
// array of octrees).  Pure integer work: every entry is found by binary
// search of the Morton keys of the sorted leaves.
#include "cello_internal.h"
#include "morton.h"

namespace cello {

// Index of the leaf whose key equals `key`, or -1.
__device__ __forceinline__ int find_key(const unsigned long long* keys, int B, unsigned long long key) {
  int lo = 0, hi = B;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (keys[mid] < key) lo = mid + 1;
    else hi = mid;
  }
  return (lo < B && keys[lo] == key) ? lo : -1;
}

// face: the kinds of the six faces of each leaf once more, in register order
// (-x, +x, -y, +y, -z, +z); bad: bit 0 a neighbour two levels coarser, bit 1 a
// child of a refined neighbour that touches the leaf is not a leaf.
__global__ void neighbour_kernel(DevMesh m, const unsigned long long* keys, int8_t* kind, int* idx, int* fine8,
                                 int8_t* face, int* bad) {
  const long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= (long)m.B * 27) return;
  const int b = (int)(gid / 27), e = (int)(gid % 27);
  const int dx = e % 3 - 1, dy = (e / 3) % 3 - 1, dz = e / 9 - 1;
  const int4 lf = m.leaf[b];
  const int L = lf.x;
  int node[3] = {lf.y + dx, lf.z + dy, lf.w + dz};
  int8_t k = kBoundary;
  int id = -1;
  int f8[8] = {-1, -1, -1, -1, -1, -1, -1, -1};
  bool inside = true;
  for (int a = 0; a < 3; ++a) {
    const int nb = m.root[a] << L;
    if (node[a] < 0 || node[a] >= nb) {
      if (m.bc[a] == 0) node[a] = (node[a] % nb + nb) % nb;
      else inside = false;
    }
  }
  if (inside) {
    const int sh = m.max_level - L;
    const int pos = find_key(keys, m.B, morton3((unsigned)node[0] << sh, (unsigned)node[1] << sh,
                                                (unsigned)node[2] << sh));
    const int plev = pos >= 0 ? m.leaf[pos].x : -1;
    if (pos >= 0 && plev == L) {
      k = kSame;
      id = pos;
    } else if (pos >= 0 && plev > L) {
      k = kFine;
      const int s1 = sh - 1;
      bool missing = false;
      for (int o = 0; o < 8; ++o) {
        const int ox = o & 1, oy = (o >> 1) & 1, oz = o >> 2;
        const unsigned cx = 2u * node[0] + ox, cy = 2u * node[1] + oy, cz = 2u * node[2] + oz;
        const int c = find_key(keys, m.B, morton3(cx << s1, cy << s1, cz << s1));
        f8[o] = (c >= 0 && m.leaf[c].x == L + 1) ? c : -1;
        // the refresh and the slope lookups index only the children that touch the leaf
        const bool apart = (dx == 1 && ox) || (dx == -1 && !ox) || (dy == 1 && oy) || (dy == -1 && !oy) ||
                           (dz == 1 && oz) || (dz == -1 && !oz);
        missing = missing || (!apart && f8[o] < 0);
      }
      if (missing) atomicOr(bad, 2);
    } else {
      const int s1 = sh + 1;
      const int c = find_key(keys, m.B, morton3((unsigned)(node[0] >> 1) << s1, (unsigned)(node[1] >> 1) << s1,
                                                (unsigned)(node[2] >> 1) << s1));
      if (c >= 0 && m.leaf[c].x == L - 1) {
        k = kCoarse;
        id = c;
      } else {
        k = -1;  // broken balance: reported by the host
        atomicOr(bad, 1);
      }
    }
  }
  kind[gid] = k;
  const int side = dx + dy + dz;   // of a face direction
  if (dx * dx + dy * dy + dz * dz == 1) face[b * 6 + 2 * (dy ? 1 : (dz ? 2 : 0)) + (side > 0 ? 1 : 0)] = k;
  idx[gid] = id;
  for (int o = 0; o < 8; ++o) fine8[gid * 8 + o] = f8[o];
}

void launch_neighbour_table(const DevMesh& m, const unsigned long long* keys, int8_t* kind, int* idx, int* fine8,
                            int8_t* face, int* bad, cudaStream_t s) {
  const long threads = (long)m.B * 27;
  if (threads <= 0) return;
  neighbour_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(m, keys, kind, idx, fine8, face, bad);
}

// Register slots of the four fine faces behind each coarse face.
__global__ void fine_slots_kernel(DevMesh m, CoarseFace* faces, int count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count * 4) return;
  CoarseFace& cf = faces[i >> 2];
  const int o1 = i & 1, o2 = (i >> 1) & 1;
  const int t1 = cf.axis == 0 ? 1 : 0, t2 = cf.axis == 2 ? 1 : 2;
  int o[3];
  o[cf.axis] = cf.side < 0 ? 1 : 0;
  o[t1] = o1;
  o[t2] = o2;
  const int e = cf.leaf * 27 + face_dir(cf.axis, cf.side);
  const int c = m.fine8[e * 8 + o[2] * 4 + o[1] * 2 + o[0]];
  cf.fslot[o2 * 2 + o1] = m.face_slot[c * 6 + 2 * cf.axis + (cf.side < 0 ? 1 : 0)];
}

void launch_fine_slots(const DevMesh& m, CoarseFace* faces, int count, cudaStream_t s) {
  fine_slots_kernel<<<(unsigned)((count * 4 + 127) / 128), 128, 0, s>>>(m, faces, count);
}

// The source of each new leaf's cells in the old mesh: the same leaf, the coarser
// leaf that contains it, or its eight children; bad is set where there is none.
__global__ void remap_map_kernel(DevMesh neu, const unsigned long long* nkeys, DevMesh old,
                                 const unsigned long long* okeys, RemapEntry* map, int* bad) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= neu.B) return;
  const int4 t = neu.leaf[b];
  int lo = 0, hi = old.B;   // the last old leaf whose key does not exceed this leaf's
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (okeys[mid] <= nkeys[b]) lo = mid + 1;
    else hi = mid;
  }
  RemapEntry e = {};
  bool found = false;
  if (lo > 0) {
    const int4 a = old.leaf[lo - 1];
    const int k = t.x - a.x;
    if (k >= 0 && (t.y >> k) == a.y && (t.z >> k) == a.z && (t.w >> k) == a.w) {
      e.kind = k == 0 ? 0 : 1;
      e.k = k;
      e.src[0] = lo - 1;
      found = true;
    }
  }
  if (!found && t.x < neu.max_level) {
    e.kind = 2;
    found = true;
    const int s1 = neu.max_level - t.x - 1;
    for (int o = 0; o < 8; ++o) {
      const unsigned cx = 2u * t.y + (o & 1), cy = 2u * t.z + ((o >> 1) & 1), cz = 2u * t.w + (o >> 2);
      const int c = find_key(okeys, old.B, morton3(cx << s1, cy << s1, cz << s1));
      if (c >= 0 && old.leaf[c].x == t.x + 1) e.src[o] = c;
      else found = false;
    }
  }
  if (!found) atomicOr(bad, 1);
  map[b] = e;
}

void launch_remap_map(const DevMesh& neu, const unsigned long long* nkeys, const DevMesh& old,
                      const unsigned long long* okeys, RemapEntry* map, int* bad, cudaStream_t s) {
  remap_map_kernel<<<(unsigned)((neu.B + 127) / 128), 128, 0, s>>>(neu, nkeys, old, okeys, map, bad);
}

}  // namespace cello
