"""The host side's compiled forms, built on their own with address and
undefined-behaviour checks: an expansion and the run after it as one bit-sliced
pass, over phase counts around every limit of that form."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2105_01533_gb300", "csrc")

EXPAND = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "sps_internal.h"
using namespace sps;
static sps_gate gate(uint8_t op, uint16_t t, int c, double th) {
  sps_gate g;
  std::memset(&g, 0, sizeof(g));
  g.op = op;
  g.t0 = t;
  if (c >= 0) g.cmask[c >> 6] = 1ull << (c & 63);
  g.theta = th;
  return g;
}
// argv: head gates, their op, controlled Rz, controlled P, T gates
int main(int, char** v) {
  const int head = std::atoi(v[1]), op = std::atoi(v[2]), nrz = std::atoi(v[3]), np = std::atoi(v[4]),
            nt = std::atoi(v[5]);
  const uint32_t nq = 60;
  std::vector<sps_gate> g;
  for (int q = 0; q < head; ++q) g.push_back(gate(op, q, -1, 1.2 + 0.01 * q));
  for (int q = 0; q < head; ++q) g.push_back(gate(SPS_OP_X, 24 + q, q, 0.0));
  for (int k = 0; k < nrz; ++k) g.push_back(gate(SPS_OP_RZ, k % head, (k + 1) % head, 0.1 + k));
  for (int k = 0; k < np; ++k) g.push_back(gate(SPS_OP_P, k % head, (k + 1) % head, 0.1 + k));
  for (int k = 0; k < nt; ++k) g.push_back(gate(SPS_OP_T, k % head, -1, 0.0));
  std::vector<Pass> p;
  KnownBits kb;
  kb.known[0] = (1ull << nq) - 1;
  size_t bad = 0;
  if (compile(g.data(), g.size(), nq, 0, &p, &bad, &kb, true, true, 4, false) != SPS_OK) return 2;
  if (p.size() < 2 || p[0].kind != PASS_EXPAND || p[1].kind != PASS_FUSED) return 3;
  BsPass run;
  build_bitslice(p[1], nq, &run);
  BsPass* b = new BsPass;
  const bool ok = build_bitslice_expand(p[0], p[1], nq, 1e-14, b);
  uint32_t bits = 0;
  for (uint32_t c = 0; ok && c < b->nchunks; ++c) bits += b->chunk_bits[c];
  std::printf("%u %d %u %u %u %d\n", run.aux_bits, ok ? 1 : 0, ok ? b->aux_bits : 0u,
              ok ? b->nchunks : 0u, bits, ok && b->direct ? 1 : 0);
  delete b;
  return 0;
}
"""


def built(tmp, name, source):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    src, exe = str(tmp / (name + ".cpp")), str(tmp / name)
    with open(src, "w") as f:
        f.write(source)
    subprocess.run([cxx, "-std=c++17", "-O1", "-g", "-fsanitize=address,undefined",
                    "-fno-sanitize-recover=all", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC,
                    src, os.path.join(CSRC, "sps_compile.cpp"), "-o", exe], check=True)
    return exe


@pytest.fixture(scope="module")
def expand(tmp_path_factory):
    return built(tmp_path_factory.mktemp("forms"), "expand", EXPAND)


@pytest.mark.parametrize("head,op,nrz,np,nt", [
    # rotations (two factors each) before the run's phases: one table of 22 bits at most
    (5, "ry", 0, 12, 0), (5, "ry", 0, 13, 0), (4, "rx", 5, 1, 3), (4, "rx", 5, 2, 3),
    (20, "ry", 16, 0, 0), (20, "ry", 17, 0, 0), (20, "ry", 28, 0, 0), (24, "ry", 30, 0, 1),
    (24, "rx", 30, 1, 1),
    # Hadamards: the run's phases alone, up to 64 bits in four tables
    (20, "h", 11, 0, 0), (20, "h", 10, 0, 3), (20, "h", 18, 0, 0), (20, "h", 27, 0, 0),
    (20, "h", 30, 1, 0), (20, "h", 30, 1, 1)])
def test_expansion_and_run_within_their_tables(expand, head, op, nrz, np, nt):
    code = {"h": 10, "rx": 11, "ry": 12}[op]
    r = subprocess.run([expand] + [str(x) for x in (head, code, nrz, np, nt)], capture_output=True,
                       text=True)
    assert r.returncode == 0, r.stderr
    run_aux, ok, aux, nchunks, bits, direct = (int(x) for x in r.stdout.split())
    assert run_aux == 2 * nrz + np + (3 if nt else 0)
    want = run_aux + (0 if op == "h" else 2 * head)
    assert ok == (want <= (64 if op == "h" else 22))
    if ok:
        assert aux == want == bits and direct == (want <= 22) and nchunks <= 4


STREAM = r"""
#include <cstdio>
#include <cstring>
#include "sps_internal.h"
using namespace sps;
// The longest op stream over runs of 512 ops: dependent Y gates, Y gates on all
// qubits, Rz and Y in turn, ladders, and random gates with up to 3 controls.
int main() {
  unsigned long long seed = 7, longest = 0;
  auto below = [&](unsigned n) {
    seed = seed * 6364136223846793005ull + 1442695040888963407ull;
    return (unsigned)((seed >> 33) % n);
  };
  for (uint32_t nq : {3u, 24u, 63u, 64u, 100u, 127u})
    for (int form = 0; form < 12; ++form) {
      std::vector<sps_gate> g;
      for (int i = 0; i < 600; ++i) {
        sps_gate r;
        std::memset(&r, 0, sizeof(r));
        auto ctl = [&](uint32_t q) { if (q != r.t0) r.cmask[q >> 6] |= 1ull << (q & 63); };
        r.op = SPS_OP_Y;
        r.t0 = form == 0 ? (uint16_t)(nq - 1) : (uint16_t)(i % nq);
        r.theta = 0.3;
        if (form == 2 && i % 20 == 1) r.op = SPS_OP_RZ;
        if (form == 2) r.t0 = (uint16_t)(nq - 1);
        if (form == 3) { r.op = SPS_OP_X; ctl((i + nq - 1) % nq); }
        if (form == 4) ctl((i + nq - 1) % nq);
        if (form > 4) {
          const uint8_t ops[] = {SPS_OP_X, SPS_OP_Y, SPS_OP_T, SPS_OP_S, SPS_OP_Y, SPS_OP_Z};
          r.op = ops[below(6)];
          r.t0 = (uint16_t)below(form > 8 ? 3 : nq);
          for (unsigned c = below(4); c; --c) ctl(below(form > 8 ? 3 : nq));
        }
        g.push_back(r);
      }
      std::vector<Pass> p;
      size_t bad = 0;
      if (compile(g.data(), g.size(), nq, 0, &p, &bad) != SPS_OK) return 2;
      for (const Pass& q : p) {
        if (q.kind != PASS_FUSED || q.ops.size() > kMaxFusedOps) return 3;
        if (q.words.size() * sizeof(OpWord) > longest) longest = q.words.size() * sizeof(OpWord);
      }
    }
  std::printf("%llu %u %u\n", longest, (unsigned)kMaxOpStreamBytes, (unsigned)kDefaultSmemBytes);
  return 0;
}
"""


def test_op_streams_within_their_limit(tmp_path):
    """Every launch that walks an op stream asks for one limit, the longest
    stream's; streams past the default of 48 KB do occur."""
    out = subprocess.run([built(tmp_path, "stream", STREAM)], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    longest, most, default = (int(x) for x in out.stdout.split())
    assert default < longest <= most
    # with the largest static shared memory of those kernels (48 KB) in an SM's 227 KB
    assert most + default <= 227 * 1024


OCCUPANCY = r"""
#include <cstdio>
#include <thread>
#include "sps_internal.h"
using namespace sps;
static int kernel_a() { return 5; }
static int kernel_b() { return 3; }
template <int (*K)()>
static int ask(int threads, size_t smem, int* queries) {
  return cached_occupancy<K>(threads, smem, [&] { ++*queries; return smem > 100000 ? 0 : K() + threads / 128; });
}
int main() {
  int q = 0;
  if (ask<kernel_a>(128, 64, &q) != 6 || ask<kernel_b>(128, 64, &q) != 4) return 2;
  if (ask<kernel_a>(128, 64, &q) != 6 || q != 2) return 3;          // kept, each its own
  if (ask<kernel_a>(256, 64, &q) != 7 || ask<kernel_a>(256, 80, &q) != 7 || q != 4) return 4;
  if (ask<kernel_a>(256, 200000, &q) != 0 || ask<kernel_a>(256, 200000, &q) != 0 || q != 6) return 5;
  bool bad[2] = {false, false};
  auto work = [&](int t) {
    int n = 0;
    for (int i = 0; i < 200000; ++i) {
      const int threads = (i + t) & 1 ? 128 : 256;
      if (ask<kernel_b>(threads, 16 * (size_t)t, &n) != 3 + threads / 128) bad[t] = true;
    }
  };
  std::thread other(work, 1);
  work(0);
  other.join();
  return bad[0] || bad[1] ? 6 : 0;
}
"""


def test_occupancy_kept_per_kernel_instance(tmp_path):
    """Instances of one type, other block sizes and shared memory, failures, and
    two threads: an answer is never another question's."""
    assert subprocess.run([built(tmp_path, "occupancy", OCCUPANCY)]).returncode == 0


WRITES = r"""
#include "sps_internal.h"
using namespace sps;
int main() {
  const uintptr_t a = 0x7f0000001000;
  struct { MemKind kind; int owner, device, current; uintptr_t at; bool host_too, want; } t[] = {
      {MEM_DEVICE, 0, 0, 0, a, false, true},  {MEM_DEVICE, 0, 0, 0, a + 8, true, true},
      {MEM_DEVICE, 1, 1, 1, a, false, true},  {MEM_PINNED, 0, 0, 0, a, true, true},
      {MEM_PINNED, 1, 0, 0, a, true, true},                       // pinned for every device
      {MEM_DEVICE, 0, 0, 1, a, false, false},                     // another device is current
      {MEM_PINNED, 0, 0, 1, a, true, false},  {MEM_DEVICE, 1, 0, 0, a, false, false},
      {MEM_DEVICE, 1, 0, 1, a, false, false}, {MEM_PINNED, 0, 0, 0, a, false, false},
      {MEM_OTHER, 0, 0, 0, a, true, false},   {MEM_DEVICE, 0, 0, 0, a + 4, false, false},
      {MEM_DEVICE, 0, 0, 0, 0, false, false}, {MEM_DEVICE, 0, 0, -1, a, false, false},
  };
  for (const auto& c : t)
    if (kernel_may_write(c.kind, c.owner, c.device, c.current, c.at, c.host_too) != c.want) return 1;
  return 0;
}
"""


def test_who_writes_the_callers_memory(tmp_path):
    """A read-back or readout goes by kernel only where a kernel can be launched and
    can write: else by copies, as with another device current."""
    assert subprocess.run([built(tmp_path, "writes", WRITES)]).returncode == 0


WALK = r"""
#include <cstdio>
#include <cstring>
#include "sps_internal.h"
using namespace sps;
typedef unsigned long long u64;
static u64 seed = 11;
static u64 rnd() {
  seed = seed * 6364136223846793005ull + 1442695040888963407ull;
  u64 x = seed;
  x ^= x >> 31;
  return x * 0x9E3779B97F4A7C15ull;
}
static unsigned below(unsigned n) { return (unsigned)((rnd() >> 33) % n); }
struct Label { u64 k[2]; unsigned cnt; u64 fire; };
// the ops in order: pi/4 steps and the slots of the phases that apply, as met
static void direct(const Pass& p, Label& l) {
  unsigned slot = 0;
  for (const FOp& o : p.ops) {
    const unsigned s0 = slot, s1 = slot + 1;
    if (o.ph != NO_PH) slot += o.sbit != NO_SEL ? 2 : 1;
    if ((l.k[0] & o.c[0]) != o.c[0] || (l.k[1] & o.c[1]) != o.c[1]) continue;
    const bool sel = o.sbit != NO_SEL && ((l.k[o.sbit >> 6] >> (o.sbit & 63)) & 1ull);
    l.cnt += sel ? o.a1 : o.a0;
    if (o.ph != NO_PH) l.fire |= 1ull << (sel ? s1 : s0);
    l.k[0] ^= o.t[0];
    l.k[1] ^= o.t[1];
  }
  l.cnt &= 7u;
}
static u64 forms[6];
static void stream(const Pass& p, Label& l) {
  if (p.words.empty()) return;
  const OpWord* W = p.words.data();
  const uint32_t* runs = &W[1].x;
  size_t q = W[0].y;
  u64 ph = 0;
  auto holds = [&](u64 c0, u64 c1) { return (l.k[0] & c0) == c0 && (l.k[1] & c1) == c1; };
  auto two = [](uint32_t a, uint32_t b) { return (u64)b << 32 | a; };
  for (uint32_t r = 0; r < W[0].x; ++r) {
    const uint32_t run = runs[r], n = run & 0xFFFFu, np = (run >> 16) & 0x1FFFu;
    const bool wide = run & kRunWide, any = run & kRunAny;
    const int S = wide ? 2 : 1;
    forms[(wide ? 3 : 0) + (run & kRunSingle ? (any ? 2 : 1) : 0)] += 1;
    if (run & kRunSingle) {
      for (uint32_t k = 0; k < n; ++k, q += S + (any ? 1 : 0)) {
        if (!holds(two(W[q].x, W[q].y), wide ? two(W[q].z, W[q].w) : 0)) continue;
        const OpWord t = wide ? W[q + 1] : OpWord{W[q].z, W[q].w, 0, 0};
        l.k[0] ^= two(t.x, t.y);
        l.k[1] ^= two(t.z, t.w);
        if (any) ph += two(W[q + S].x, W[q + S].y);
      }
      continue;
    }
    for (uint32_t k = 0; k < n + np; ++k) {   // both conditions on the label before the step
      bool on[2];
      OpWord t[2];
      for (int h = 0; h < 2; ++h, q += S) {
        on[h] = holds(two(W[q].x, W[q].y), wide ? two(W[q].z, W[q].w) : 0);
        t[h] = wide ? W[q + 1] : OpWord{W[q].z, W[q].w, 0, 0};
      }
      for (int h = 0; h < 2; ++h)
        if (on[h]) {
          if (k < n) {
            l.k[0] ^= two(t[h].x, t[h].y);
            l.k[1] ^= two(t[h].z, t[h].w);
          } else {
            ph += two(t[h].x, t[h].y);
          }
        }
    }
  }
  if (q + 4 != p.words.size()) std::printf("length %zu of %zu\n", q, p.words.size());
  l.cnt = (unsigned)(ph >> kOpCountShift) & 7u;
  l.fire = ph & ((1ull << kOpCountShift) - 1);
}
int main() {
  int bad = 0;
  for (uint32_t nq : {2u, 5u, 24u, 63u, 64u, 70u, 127u})
    for (int round = 0; round < 220; ++round) {
      const int form = round % 11;
      std::vector<sps_gate> g;
      const int count = round % 3 == 0 ? 1 + (int)below(12) : 20 + (int)below(500);
      for (int i = 0; i < count; ++i) {
        sps_gate r;
        std::memset(&r, 0, sizeof(r));
        auto ctl = [&](uint32_t q) { if (q != r.t0) r.cmask[q >> 6] |= 1ull << (q & 63); };
        r.op = SPS_OP_X;
        r.t0 = (uint16_t)(i % nq);
        r.theta = 0.1 + i;
        const uint8_t all[] = {SPS_OP_X, SPS_OP_Y, SPS_OP_Z, SPS_OP_S, SPS_OP_TDG, SPS_OP_P, SPS_OP_RZ};
        if (form == 3) r.t0 = (uint16_t)below(3 < nq ? 3 : nq);
        if (form == 6) r.t0 = (uint16_t)below(nq);
        if (form > 6) r.t0 = (uint16_t)(form == 10 ? nq - 1 - below(2) : below(nq));
        if (form < 4) ctl((i + nq - 1) % nq);                           // ladders
        if (form == 1 && i % 3 == 1) r.op = SPS_OP_T;                  // with phases between
        if (form == 2 && i % 40 > 20) r.op = all[below(7)];
        if (form == 4) r.op = SPS_OP_Y, r.t0 = (uint16_t)(nq - 1);
        if (form == 5) { r.op = SPS_OP_Y; ctl(below(nq)); }
        if (form == 6) { ctl(below(nq)); ctl(below(nq)); }
        if (form > 6) {
          r.op = all[below(7)];
          for (unsigned c = below(form == 9 ? 7 : 3); c; --c) ctl(below(nq));
        }
        g.push_back(r);
      }
      std::vector<Pass> ps;
      size_t at = 0;
      KnownBits kb;
      if (round & 1) { kb.known[0] = rnd() & rnd(); kb.known[0] &= nq < 64 ? (1ull << nq) - 1 : ~0ull; }
      const KnownBits k0 = kb;
      if (compile(g.data(), g.size(), nq, 0, &ps, &at, round & 1 ? &kb : nullptr, false, true) != SPS_OK)
        return 2;
      for (int e = 0; e < 40; ++e) {
        Label l{{rnd(), rnd()}, 0, 0};
        l.k[0] &= nq < 64 ? (1ull << nq) - 1 : ~0ull;
        l.k[1] &= nq > 64 ? (1ull << (nq - 64)) - 1 : 0ull;
        l.k[0] &= ~k0.known[0];   // (known to be 0)
        for (const Pass& p : ps) {
          Label a = l, b = l;
          a.cnt = b.cnt = 0;
          a.fire = b.fire = 0;
          direct(p, a);
          stream(p, b);
          if (a.k[0] != b.k[0] || a.k[1] != b.k[1] || a.cnt != b.cnt || a.fire != b.fire) ++bad;
          l = a;
        }
      }
    }
  std::printf("%d %llu %llu %llu %llu %llu %llu\n", bad, forms[0], forms[1], forms[2], forms[3], forms[4], forms[5]);
  return bad != 0;
}
"""


def test_op_streams_do_what_their_ops_do(tmp_path):
    """Every form of run, on labels of both widths, with and without known qubits:
    the stream's flips, pi/4 steps and phase slots against the ops one by one."""
    out = subprocess.run([built(tmp_path, "walk", WALK)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    words = [int(x) for x in out.stdout.split()]
    assert words[0] == 0 and min(words[1:]) > 0, words


LENGTHS = r"""
#include <cstdio>
#include <cstring>
#include "sps_internal.h"
using namespace sps;
// words and pairs of flips of the streams of: a CNOT ladder, Y gates on one qubit,
// CNOTs on 24 disjoint pairs
int main() {
  for (int form = 0; form < 3; ++form) {
    std::vector<sps_gate> g;
    auto cx = [&](int a, int b, int t) {
      sps_gate r;
      std::memset(&r, 0, sizeof(r));
      r.op = SPS_OP_X;
      r.t0 = (uint16_t)t;
      r.cmask[0] = (a >= 0 ? 1ull << a : 0ull) | (b >= 0 ? 1ull << b : 0ull);
      g.push_back(r);
    };
    for (int i = 0; form == 0 && i < 480; ++i) cx(i % 48, -1, (i + 1) % 48);
    for (int i = 0; form == 1 && i < 480; ++i) {
      cx(-1, -1, 3);
      g.back().op = SPS_OP_Y;
    }
    for (int i = 0; form == 2 && i < 480; ++i) cx(2 * (i % 24), -1, 2 * (i % 24) + 1);
    std::vector<Pass> p;
    size_t bad = 0;
    if (compile(g.data(), g.size(), 50, 0, &p, &bad) != SPS_OK || p.size() != 1) return 2;
    uint32_t pairs = 0;
    for (uint32_t r = 0; r < p[0].words[0].x; ++r)
      pairs += (&p[0].words[1].x)[r] & kRunSingle ? 0u : (&p[0].words[1].x)[r] & 0xFFFFu;
    std::printf("%zu %u\n", p[0].words.size() - p[0].words[0].y - 4, pairs);
  }
  return 0;
}
"""


def test_no_half_empty_pairs_on_serial_chains(tmp_path):
    """A chain of flips that each read what the last one flipped is single steps, a
    word a flip (as pairs it would be two); flips that wait for nothing are pairs."""
    out = subprocess.run([built(tmp_path, "lengths", LENGTHS)], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    ladder, ys, disjoint = ([int(x) for x in line.split()] for line in out.stdout.splitlines())
    assert ladder == [480, 0] and disjoint == [480, 240]
    assert ys[1] <= 1   # beside the phase ops that read nothing
