// Runs one thread block of the generated kernels on the CPU: a fiber per lane, and a scheduler that lets
// the lanes of one end of the block run as far ahead of the others as the barriers and warp-level
// collectives allow (the lowest lanes with order = +1, the highest with -1).  A missing barrier
// then gives wrong numbers every time instead of once in a while, and a collective that names lanes
// which never come to it leaves the block stuck, which is reported.
//
// Included ahead of a generated source (which holds the inline PTX as calls of emu_* functions, see
// emulated.py); FX_HOST selects the host forms of the integer helpers.
#pragma once
#include <ucontext.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <vector>

namespace emu {

struct Wait {
  int kind = 0;  // 0 running, 1 block barrier, 2 warp collective, 3 exited
  int id = 0;    // barrier number, or the collective's kind
  unsigned mask = 0, count = 0;
  uint64_t in[16] = {};
  std::vector<uint64_t> out;  // a collective's inputs of all 32 lanes
  bool flag = false, any = false;
};

struct Block {
  int n = 0, order = 1, cur = -1;
  std::vector<Wait> w;
  std::vector<ucontext_t> ctx;
  std::vector<std::vector<char>> stack;
  ucontext_t main;
  std::function<void()> body;
};
inline Block* B = nullptr;

inline void entry() {
  B->body();
  B->w[B->cur].kind = 3;
  swapcontext(&B->ctx[B->cur], &B->main);
}
inline void yield() { swapcontext(&B->ctx[B->cur], &B->main); }

// releases what is complete; returns false if nothing can run
inline void release() {
  for (int t = 0; t < B->n; ++t) {
    Wait& a = B->w[t];
    if (a.kind == 1) {
      int here = 0;
      bool any = false;
      for (auto& x : B->w)
        if ((x.kind == 1 && x.id == a.id) || (x.kind == 3 && a.id == 0)) { ++here; any = any || (x.kind == 1 && x.flag); }
      if (here < (int)a.count) continue;
      for (auto& x : B->w)
        if (x.kind == 1 && x.id == a.id) { x.kind = 0; x.any = any; }
    } else if (a.kind == 2) {
      const int w0 = t / 32 * 32;
      bool all = true;
      for (int l = 0; l < 32 && all; ++l)
        if (a.mask >> l & 1) {
          const Wait* x = w0 + l < B->n ? &B->w[w0 + l] : nullptr;
          all = x && x->kind == 2 && x->id == a.id && x->mask == a.mask;
        }
      if (!all) continue;
      std::vector<uint64_t> out(32 * 16);
      for (int l = 0; l < 32 && w0 + l < B->n; ++l)
        if (a.mask >> l & 1) memcpy(&out[l * 16], B->w[w0 + l].in, sizeof(a.in));
      const unsigned mask = a.mask;
      for (int l = 0; l < 32; ++l)
        if (mask >> l & 1) { B->w[w0 + l].out = out; B->w[w0 + l].kind = 0; }
    }
  }
}

// one block of n lanes; returns false (with a message) if lanes wait for others that never come
inline bool run(int n, int order, std::function<void()> body) {
  Block blk;
  B = &blk;
  blk.n = n;
  blk.order = order;
  blk.body = body;
  blk.w.resize(n);
  blk.ctx.resize(n);
  blk.stack.assign(n, std::vector<char>(256 << 10));
  for (int t = 0; t < n; ++t) {
    getcontext(&blk.ctx[t]);
    blk.ctx[t].uc_stack.ss_sp = blk.stack[t].data();
    blk.ctx[t].uc_stack.ss_size = blk.stack[t].size();
    blk.ctx[t].uc_link = &blk.main;
    makecontext(&blk.ctx[t], entry, 0);
  }
  for (;;) {
    int next = -1, done = 0;
    for (int pass = 0; pass < 2 && next < 0; ++pass) {
      if (pass) release();
      done = 0;
      for (int i = 0; i < n && next < 0; ++i) {
        const int t = order > 0 ? i : n - 1 - i;
        if (blk.w[t].kind == 0) next = t;
        done += blk.w[t].kind == 3;
      }
    }
    if (next < 0) {
      if (done == n) return true;
      for (int t = 0; t < n; ++t)
        if (blk.w[t].kind != 3)
          fprintf(stderr, "lane %d waits at %s %d (mask %08x)\n", t, blk.w[t].kind == 1 ? "barrier" : "collective",
                  blk.w[t].id, blk.w[t].mask);
      return false;
    }
    blk.cur = next;
    swapcontext(&blk.main, &blk.ctx[next]);
    release();  // a lane whose partners have all come goes on before lanes behind it in the order
  }
}

inline bool barrier(int id, int count, bool flag = false) {
  Wait& w = B->w[B->cur];
  w.kind = 1;
  w.id = id;
  w.count = (unsigned)count;
  w.flag = flag;
  yield();
  return B->w[B->cur].any;
}

enum { SYNC, ANY, RMAX, RMIN, SHFL, MMA16, MMA8 };
inline const uint64_t* collect(int kind, unsigned mask, const uint64_t* in, int n) {
  Wait& w = B->w[B->cur];
  if (!(mask >> (B->cur & 31) & 1)) { fprintf(stderr, "lane %d is not in its own mask\n", B->cur); exit(3); }
  w.kind = 2;
  w.id = kind;
  w.mask = mask;
  std::copy(in, in + n, w.in);
  yield();
  return B->w[B->cur].out.data();
}
template <class T>
T get(const uint64_t* o, int lane, int i = 0) { T v; memcpy(&v, &o[lane * 16 + i], sizeof(T)); return v; }
template <class T>
T shfl(unsigned mask, T v, int src) {
  uint64_t b = 0;
  memcpy(&b, &v, sizeof(T));
  const uint64_t* o = collect(SHFL, mask, &b, 1);
  if (!(mask >> src & 1)) { fprintf(stderr, "shuffle from lane %d outside the mask\n", src); exit(3); }
  return get<T>(o, src);
}
inline int lane() { return B->cur & 31; }

inline float half(unsigned h) {
  const int e = (h >> 10) & 31, m = h & 1023;
  const float v = e ? std::ldexp(1024.0f + m, e - 25) : std::ldexp((float)m, -24);
  return h & 0x8000 ? -v : v;
}
inline unsigned to_half(float v) {  // exact values only
  if (v == 0) return 0;
  int e;
  const float m = std::frexp(std::fabs(v), &e);
  return (v < 0 ? 0x8000u : 0u) | (unsigned)(e + 14) << 10 | ((unsigned)std::ldexp(m, 11) & 1023u);
}
// D += A B for an m16n8 tile with k = 16 (na = 4, nb = 2 registers) or 8 (2, 1)
inline void mma(int kind, float* c, const unsigned* a, int na, const unsigned* b, int nb) {
  uint64_t in[6];
  for (int i = 0; i < na; ++i) in[i] = a[i];
  for (int i = 0; i < nb; ++i) in[na + i] = b[i];
  const uint64_t* o = collect(kind, 0xffffffffu, in, na + nb);
  const int g = lane() >> 2, t = lane() & 3;
  for (int i = 0; i < 4; ++i) {
    const int r = g + (i >= 2 ? 8 : 0), n = 2 * t + (i & 1);
    double s = c[i];
    for (int k = 0; k < 8 * nb; ++k) {
      const unsigned ra = (unsigned)o[((r & 7) * 4 + (k & 7) / 2) * 16 + (r >= 8) + (k >= 8 ? 2 : 0)];
      const unsigned rb = (unsigned)o[(n * 4 + (k & 7) / 2) * 16 + na + (k >= 8)];
      s += (double)half(k & 1 ? ra >> 16 : ra & 0xffff) * half(k & 1 ? rb >> 16 : rb & 0xffff);
    }
    c[i] = (float)s;
  }
}

struct Dim { unsigned x; };
}  // namespace emu

// ---- the CUDA names that the generated source uses
using std::isfinite;
using std::max;
using std::min;
#define __device__
#define __global__
#define __shared__
#define __forceinline__ inline
#define __noinline__ __attribute__((noinline))
#define __launch_bounds__(...)
#define __align__(n) __attribute__((aligned(n)))
#define threadIdx (emu::Dim{(unsigned)emu::B->cur})
#define blockDim (emu::Dim{(unsigned)emu::B->n})
#define blockIdx (emu::Dim{0u})
#define gridDim (emu::Dim{1u})
struct alignas(16) uint4 { unsigned x, y, z, w; };
struct alignas(16) int4 { int x, y, z, w; };
struct alignas(16) longlong2 { long long x, y; };
inline uint4 make_uint4(unsigned x, unsigned y, unsigned z, unsigned w) { return {x, y, z, w}; }
inline long long __double_as_longlong(double d) { long long v; memcpy(&v, &d, 8); return v; }
inline double __longlong_as_double(long long v) { double d; memcpy(&d, &v, 8); return d; }
inline unsigned __float_as_uint(float f) { unsigned v; memcpy(&v, &f, 4); return v; }
inline void __syncthreads() { emu::barrier(0, emu::B->n); }
inline int __syncthreads_or(int f) { return emu::barrier(0, emu::B->n, f != 0); }
inline void emu_bar(int id, int n) { emu::barrier(id, n); }
inline void __syncwarp(unsigned m = 0xffffffffu) { uint64_t z = 0; emu::collect(emu::SYNC, m, &z, 1); }
inline bool __any_sync(unsigned m, bool f) {
  uint64_t v = f;
  const uint64_t* o = emu::collect(emu::ANY, m, &v, 1);
  for (int l = 0; l < 32; ++l) if ((m >> l & 1) && o[l * 16]) return true;
  return false;
}
inline unsigned __reduce_max_sync(unsigned m, unsigned v) {
  uint64_t b = v;
  const uint64_t* o = emu::collect(emu::RMAX, m, &b, 1);
  unsigned r = 0;
  for (int l = 0; l < 32; ++l) if (m >> l & 1) r = max(r, (unsigned)o[l * 16]);
  return r;
}
inline unsigned __reduce_min_sync(unsigned m, unsigned v) {
  uint64_t b = v;
  const uint64_t* o = emu::collect(emu::RMIN, m, &b, 1);
  unsigned r = ~0u;
  for (int l = 0; l < 32; ++l) if (m >> l & 1) r = min(r, (unsigned)o[l * 16]);
  return r;
}
template <class T> T __shfl_sync(unsigned m, T v, int src, int w = 32) {
  const int base = emu::lane() / w * w;
  return emu::shfl(m, v, base + (src & (w - 1)));
}
template <class T> T __shfl_xor_sync(unsigned m, T v, int o) { return emu::shfl(m, v, emu::lane() ^ o); }
template <class T> T __shfl_down_sync(unsigned m, T v, int o, int w = 32) {
  const int l = emu::lane(), base = l / w * w;
  return emu::shfl(m, v, l - base + o < w ? l + o : l);
}
template <class T> T atomicAdd(T* p, T v) { const T old = *p; *p = old + v; return old; }
inline int atomicMax(int* p, int v) { const int old = *p; *p = max(old, v); return old; }
inline unsigned emu_hsub2(unsigned a, unsigned b) {
  return emu::to_half(emu::half(a & 0xffff) - emu::half(b & 0xffff)) |
         emu::to_half(emu::half(a >> 16) - emu::half(b >> 16)) << 16;
}
inline void emu_mma16(float* c, unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
  const unsigned a[4] = {a0, a1, a2, a3}, b[2] = {b0, b1};
  emu::mma(emu::MMA16, c, a, 4, b, 2);
}
inline void emu_mma8(float* c, unsigned a0, unsigned a1, unsigned b0) {
  const unsigned a[2] = {a0, a1}, b[1] = {b0};
  emu::mma(emu::MMA8, c, a, 2, b, 1);
}
#define FX_HOST
#define FX_FN static inline
#define FX_SLOW static
#define FX_TAB static const
typedef unsigned long long fx_u64;
typedef long long fx_i64;
FX_FN fx_u64 fx_mulhi(fx_u64 a, fx_u64 b) { return (fx_u64)(((unsigned __int128)a * b) >> 64); }
FX_FN fx_i64 fx_mulhi_s(fx_i64 a, fx_i64 b) { return (fx_i64)(((__int128)a * b) >> 64); }
FX_FN unsigned fx_mulhi32(unsigned a, unsigned b) { return (unsigned)(((fx_u64)a * b) >> 32); }
FX_FN int fx_mulhi32_s(int a, int b) { return (int)(((fx_i64)a * b) >> 32); }
FX_FN int fx_clz(fx_u64 a) { return a ? __builtin_clzll(a) : 64; }
FX_FN double fx_as_double(fx_u64 a) { double d; memcpy(&d, &a, 8); return d; }
FX_FN fx_u64 fx_bits(double a) { fx_u64 d; memcpy(&d, &a, 8); return d; }
FX_FN float fx_rcp_seed(float f) { return 1.0f / f; }
FX_FN unsigned fx_bits_f(float a) { return __float_as_uint(a); }
FX_FN float fx_as_float(unsigned a) { float d; memcpy(&d, &a, 4); return d; }
