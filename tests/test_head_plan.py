"""How the per-head kernel shares an SM between heads, compiled for the host and checked without a GPU."""
import os
import subprocess

HERE = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(HERE, "paper_2505_18698_b200", "csrc", "head_plan.h")


def test_every_plan_can_be_launched(tmp_path):
    """All shapes the kernel is made for, one round and more, from one head to many turns of the GPU: at least a CTA and a warp,
    the CTAs of an SM fit its shared memory and registers, the blocks of a warp fit the bits it keeps for them."""
    src = tmp_path / "t.cpp"
    src.write_text(f"""
#include <cstdio>
#include "{HEADER}"
using namespace ma::fhead;
int main() {{
  for (int b = 9; b <= 32; ++b)
    for (int m = 9; m <= 32; ++m)
      for (int T = 1; T <= 2; ++T)
        for (int BH : {{1, 12, 74, 75, 148, 149, 160, 296, 297, 370, 371, 444, 445, 740, 768, 100000}}) {{
          Plan p;
          const bool has = plan(b, m, T, BH, 148, &p);
          if (has && !any_fits((b + 7) / 8, (m + 7) / 8)) return 1;      // (such a kernel is not compiled)
          if (has)
            printf("%d %d %d %d %d %d %d %d %zu %d %d\\n", b, m, T, BH, p.ctas, p.warps, p.bufs, p.rounds, p.smem, p.bound,
                   p.parts);
        }}
}}""")
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-o", exe, str(src)], check=True)
    seen, whole, split = set(), set(), set()
    for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines():
        b, m, T, BH, ctas, warps, bufs, rounds, smem, most, parts = map(int, line.split())
        assert 1 <= ctas <= 3 and 1 <= warps and ctas * warps <= most and 32 * warps <= 1024, line
        assert smem <= 227 * 1024 and ctas * (smem + 1024) <= 228 * 1024, line
        assert bufs in (1, 2) and -(-m // warps) <= 15, line      # (bit 31 of the parities says that a wait ran out)
        assert (rounds == 0) == (T == 1), line
        # two CTAs a head: more than 16 positions, and an SM for each of them; a CTA then has one 16-row tile of every block
        assert parts == (2 if b > 16 and 2 * BH <= 148 else 1), line
        assert parts == 1 or (ctas == 1 and bufs == 1 and -(-b // 2) <= 16), line
        if parts * BH <= 148:
            assert 2 * (smem + 1024) > 228 * 1024, line           # a CTA an SM: no second one fits
        split |= {(b, m, T)} if parts == 2 else set()
        if BH <= 148 and max(b, m) <= 16:
            assert most == 16, line                               # few heads: all the registers a warp can use
        seen.add((b, m, T))
        if smem > 226 * 1024 and BH > 148:
            whole.add((b, m))
    assert {(31, 19), (30, 19), (28, 21), (20, 28), (21, 28)} <= whole      # one CTA takes all there is
    assert len(seen) > 700 and {(17, 25, 1), (17, 25, 2), (20, 28, 1), (31, 19, 1), (32, 12, 1)} <= split
