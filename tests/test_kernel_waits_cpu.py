"""The kernels' bounded waits, as far as they can be checked without a GPU."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_0810_1648_gb300", "csrc")


def _statements():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        for part in re.split(r"[;{}]", code):
            yield os.path.basename(path), " ".join(part.split())


def test_no_lane_skips_a_vote_of_its_warp():
    """mbar_wait_warp is a vote of all lanes: whether the warp gets that far is
    not left to each lane's own look at a flag that others set meanwhile (a lane
    that saw it would leave the others in the vote)."""
    calls = [(f, s) for f, s in _statements() if "mbar_wait_warp(" in s and "bool mbar_wait_warp" not in s]
    assert len(calls) > 10
    for f, s in calls:
        before = s[: s.index("mbar_wait_warp(")]
        assert "volatile" not in before and "abort_flag" not in before, (f, s)


RING = r"""
#include "ptx.cuh"
#include <cstdio>
// An mbarrier is its count of completed phases; a wait on a parity passes where
// the current phase has the other one.
template <int N>
int check()
{
    int bad = 0;
    for (int fills = 0; fills <= 5 * N; ++fills) {
        int done[N] = {}, stage = 0;
        uint32_t phase = 0;
        for (int k = 0; k < fills; ++k) {
            ++done[stage];                        // a fill completes one phase
            if (++stage == N) { stage = 0; phase ^= 1u; }
        }
        for (int s = 0; s < N; ++s) {
            const uint32_t p = gabp::last_fill_parity(s, stage, phase);
            if ((uint32_t)(done[s] & 1) == p) ++bad;                           // landed, and waited for in vain
            if (done[s] > 0 && (uint32_t)((done[s] - 1) & 1) != p) ++bad;      // on its way, and not waited for
        }
    }
    return bad;
}
int main() { const int bad = check<1>() + check<2>() + check<4>() + check<6>(); std::printf("%d\n", bad); return bad != 0; }
"""


def test_a_producer_waits_for_the_last_fill_of_each_stage(tmp_path):
    """The parity that await_copies waits for, against a count of fills."""
    from paper_0810_1648_gb300 import build
    src, exe = tmp_path / "ring.cu", tmp_path / "ring"
    src.write_text(RING)
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", build.INCLUDE,
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).returncode == 0


def test_every_producer_waits_for_its_copies():
    """A function that issues bulk copies ends with a wait for them, also where
    it gives up (a return after a copy has been issued)."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        copies = [m.start() for m in re.finditer(r"\bbulk_load\(", code)]
        waits = [m.start() for m in re.finditer(r"\bawait_copies<", code)]
        for c in copies:
            # before the next role of the warp-specialised kernel, or (the shared
            # producers of a sweep) within the function that issues them
            role = re.search(r"\} else if \(warp|\n\}\n", code[c:])
            begin = max(code.rfind("\n{\n", 0, c), 0)
            assert any(begin < w < c + role.end() for w in waits), (os.path.basename(path), code[c:c + 80])
