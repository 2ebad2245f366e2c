"""Blocks per SM that the shared memory of a launch configuration holds, over mechanism sizes: keeping a
chunk's rates there must not cost a resident block, or refuse a mechanism, that the layout without it
(one per-species array more) has room for, as far as the registers let the blocks be resident."""
import subprocess

from tests import emulated

MAIN = r"""
int main() {
  for (int tab = 0; tab <= 5; ++tab)
    for (int team : {4, 8, 16, 32, 64, 128, 256})
      for (int tpb : {32, 64, 128, 256})
        for (int adj = 0; adj <= (tab == 0 && team >= 32); ++adj)
          for (int mult : {2, 4, 7})
            for (int ns = 2; ns <= 170; ++ns) {
              if (check_config(team, tpb)) continue;
              const RosCoefficients c = ros_coefficients(tab);
              MechData m;
              m.sp.resize(ns);
              m.rx.resize(mult * ns);
              const int ch = chunk_size(ns, mult * ns, c, team, tpb, adj);
              if (slots_for(m, tab, team, tpb, adj) != cell_slots(ns, mult * ns, c, team, ch, false)) return 1;
              printf("%d %d %d %d %d %d %d %d\n", tab, team, tpb, adj, mult * ns, ns, ch,
                     cell_slots(ns, mult * ns, c, team, ch, adj));
            }
}
"""


def _former_slots(ns, nr, team, tab, adj):
    stages = {0: 4, 1: 3, 2: 4, 3: 6, 4: 6, 5: 3}[tab]
    f0 = 1 if tab == 2 else 0  # RODAS3 keeps f(y) for its second stage
    s = ns * ns + (8 + stages + f0) * ns + (ns + 1) // 2 + 24
    return s + (15 * ns + nr + 2 * (11 * ns + nr + 8 * team // 32) if adj else 0)


def _blocks(slots, team, tpb):
    if team < 32:
        slots += (team - slots % 16 + 16) % 16
    size = 8 * slots * max(1, tpb // team)
    return 0 if size > 227 * 1024 else 228 * 1024 // (size + 1024)


def test_chunks_cost_no_resident_block(tmp_path):
    out = subprocess.run([emulated.host_program(tmp_path, MAIN)], capture_output=True, text=True, check=True).stdout
    rows = [tuple(map(int, l.split())) for l in out.splitlines()]
    assert len(rows) > 20000
    for tab, team, tpb, adj, nr, ns, chunk, slots in rows:
        regs = 255 if adj else 128  # a thread, at most
        most = max(1, 65536 // ((regs + 1) // 8 * 8 * tpb))
        if team == 128 and ns > 64 and not adj:
            most = 2  # the kernel's register bound asks for two
        now, then = _blocks(slots, team, tpb), _blocks(_former_slots(ns, nr, team, tab, adj), team, tpb)
        assert now >= min(then, most), (tab, team, tpb, adj, nr, ns, chunk, now, then)
        assert 1 <= chunk <= min(512, nr)
    # the sizes of the three mechanisms of this repository keep their chunks
    sizes = {(r[1], r[2], r[4], r[5]): r[6] for r in rows if r[0] == 0 and not r[3]}
    assert sizes[64, 64, 7 * 53, 53] == 64 and sizes[128, 128, 7 * 53, 53] == 128 and sizes[256, 256, 7 * 111, 111] == 256
