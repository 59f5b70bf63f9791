// Host-side check of the edge candidates' records (st_device.cuh), compiled and called by test_edge_records.py.
#include "../paper_2012_03939_gb300/csrc/st_device.cuh"

// Packs a record over 48 bytes of old content (48 of `fill`) and reads it back: out = what a sample would take, the return
// value whether it would.
extern "C" int edge_round_trip(int drawable, int e, const float* f9, unsigned char fill, float* out, int* out_e) {
  float4 p[3];
  memset(p, fill, sizeof(p));
  st::EdgeRec r, q;
  if (drawable) {   // else as a clip that fails leaves it: not written
    r.sa = make_float2(f9[0], f9[1]); r.ext = make_float2(f9[2], f9[3]); r.ns = make_float2(f9[4], f9[5]);
    r.t0 = f9[6]; r.dt = f9[7]; r.len = f9[8];
    r.e = e;
  } else {
    memset(&r, fill, sizeof(r));
  }
  st::edge_pack(drawable != 0, r, p);
  const bool ok = st::edge_unpack(p[0], p[1], p[2], q);
  const float got[9] = {q.sa.x, q.sa.y, q.ext.x, q.ext.y, q.ns.x, q.ns.y, q.t0, q.dt, q.len};
  for (int k = 0; k < 9; ++k) out[k] = got[k];
  *out_e = q.e;
  return ok ? 1 : 0;
}
