"""Rules that every kernel source keeps and no GPU run can show."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_01464_gb300", "csrc")


def _code(path):
    """The source without its comments."""
    text = open(path).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("name", sorted(os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*.cu*"))))
def test_no_multicast_loads(name):
    # the library also serves one process per GPU on several GPUs, where a load
    # into several CTAs' shared memory is not to be used
    for line in re.findall(r"cp\.async\.bulk[^;]*;", _code(os.path.join(CSRC, name))):
        assert "multicast" not in line, line


def _guards(code, pos):
    """Heads of the blocks and the statement head that enclose position pos."""
    heads, depth = [], 0
    for i in range(pos - 1, -1, -1):
        if code[i] == "}":
            depth += 1
        elif code[i] == "{":
            if depth == 0:
                heads.append(code[max(code.rfind(c, 0, i) for c in ";{}") + 1:i])
            else:
                depth -= 1
    return heads + [code[max(code.rfind(c, 0, pos) for c in ";{}") + 1:pos]]


@pytest.mark.parametrize("name", ["qgemm_tc.cu", "qgemm_emu.cu", "batched_tc.cu"])
def test_no_lane_leaves_its_warp_after_a_wait(name):
    # The answer of a bounded wait is one lane's: lanes that wait together can part
    # over it (one sees the abort flag, another the barrier), and those that go on
    # would stay in elect.sync or __syncwarp for ever.  A wait is a single lane's,
    # or its answer is discarded and the warp asks warp_aborted.
    code = _code(os.path.join(CSRC, name))
    waits = [m.start() for m in re.finditer(r"mbar_wait\(", code)]
    assert len(waits) >= 4
    for pos in waits:
        guards = " ".join(_guards(code, pos))
        single = re.search(r"elect_one\(\)|lane == 0|threadIdx\.x == 0", guards)
        assert single or code[:pos].rstrip().endswith("(void)"), code[pos:pos + 60]
    issuer = open(os.path.join(CSRC, name)).read()
    issuer = issuer[issuer.index("// ---------------- MMA issuer"):]
    assert "if (warp_aborted(" in issuer[:issuer.index("// ---------------- epilogue")]
    assert re.search(r"bool warp_aborted\([^)]*\) \{\s*return __any_sync\(0xffffffffu,",
                     _code(os.path.join(CSRC, "tc_ptx.cuh")))


@pytest.mark.parametrize("name", ["qgemm_tc.cu", "qgemm_emu.cu", "batched_tc.cu"])
def test_tmem_is_freed_after_the_mmas(name):
    # A CTA that gives up may still have MMAs in flight, and their TMEM columns go
    # to the SM's next CTA: between the last block barrier of the roles and the
    # deallocation, the issuing warps wait for them.
    code = _code(os.path.join(CSRC, name))
    end = code[:code.index("tcgen05.dealloc")]
    m = re.search(r"abort_flag\) drain_mmas\(", end)
    assert m and "__syncthreads();" in end[m.end():]
    assert end[:m.start()].rfind("__syncthreads();") > end.rfind("tcgen05.alloc")


def test_waits_after_an_abort():
    # a raised flag ends a wait after few tries (an issuing warp may pass many waits
    # before its next warp_aborted), and the last wait for copies and MMAs does not
    # look at the flag
    code = _code(os.path.join(CSRC, "tc_ptx.cuh"))
    body = code[code.index("bool mbar_wait("):]
    body = body[:body.index("\n}")]
    assert re.search(r"if \(\(it & 15u\) == 0\) \{\s*if \(\*abort_flag\) return false;", body)
    drain = code[code.index("void drain_wait("):]
    drain = drain[:drain.index("\n}")]
    assert "DRAIN_NS" in drain and "abort" not in drain
    for name in ("qgemm_tc.cu", "qgemm_emu.cu", "batched_tc.cu"):
        text = _code(os.path.join(CSRC, name))
        assert re.search(r"drain_wait\(smem_u32\(&(bar_|ts\.)full\[", text), name
