"""Rules that the CUDA sources keep and that no run can show: what they forbid goes wrong on another
machine, with another compiler or under another caller's timing."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = {os.path.basename(p): open(p).read()
           for p in sorted(glob.glob(os.path.join(ROOT, "paper_2608_08569_gb300", "csrc", "*.cu*")))}
KERNELS = [(f, m.group(1), m.group(2)) for f, s in SOURCES.items()
           for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^{;]*?\)\s+)?(\w+)\s*\(([^{;]*?)\)\s*\{", s)]


def test_every_kernel_is_found():
    assert sum(len(re.findall(r"__global__", s)) for s in SOURCES.values()) == len(KERNELS) >= 10


def test_no_kernel_promises_that_its_inputs_do_not_change():
    """A programmatic dependent is resident while the kernel before it still writes: a pointer to constant
    data marked __restrict__ would allow read-only loads, which such writes must not meet."""
    bad = [(f, k, p) for f, k, params in KERNELS for p in re.findall(r"const [^,]*__restrict__ \w+", params)]
    assert not bad, bad


def test_aligned_cluster_barriers_follow_a_reconvergence():
    """The aligned forms of the cluster barrier want all lanes of a warp together. They stand in one place
    each, right after a __syncwarp()."""
    for f, s in SOURCES.items():
        lines = [x.strip() for x in s.splitlines()]
        for i, x in enumerate(lines):
            if re.search(r"barrier\.cluster\.\S*aligned", x):
                assert f == "ptx.cuh" and lines[i - 1] == "__syncwarp();", (f, i + 1)


def test_kernel_attributes_are_set_per_device():
    """An attribute belongs to a function on a device: a flag of the process would leave a second GPU without
    it (and is a race between host threads). Every setting is inside once_per_device."""
    for f, s in SOURCES.items():
        for m in re.finditer(r"cudaFuncSetAttribute\(", s):
            assert "once_per_device(" in s[max(0, m.start() - 800):m.start()], (f, s.count("\n", 0, m.start()) + 1)
        assert not re.search(r"static bool \w+", s), f


def test_decode_plans_are_kept_per_device():
    """A plan's cluster size and how many clusters are resident come from the device's occupancy."""
    s = SOURCES["decode_mma.cu"]
    assert re.search(r"struct Entry \{\s*int device\b", s) and "e.device == device" in s


def test_another_units_length_is_read_atomically():
    """The cluster of a later unit may run beside this one and store that unit's length."""
    assert not re.findall(r"p\.len\[(?!ui\.cache_unit\])", SOURCES["decode_mma.cu"])


def test_the_logits_of_a_lane_group_lie_in_different_banks():
    """Phase V of the decode reads, per lane (g, qd), head 8 nt + g of row qd + 4 e: with the row length and
    the swap of its template, no two lanes of a warp meet in a bank. The swapped column is a permutation."""
    s = SOURCES["decode_mma.cu"]
    assert "return kSwap ? h ^ ((row & 2) << 2) : h;" in s and "kSwap = NT == 2 && (kCluster || D == 64)" in s
    for heads, swap in ((8, False), (16, True)):
        col = lambda row, h: h ^ ((row & 2) << 2) if swap else h
        for row in range(16):
            assert sorted(col(row, h) for h in range(heads)) == list(range(heads))
        for nt in range(heads // 8):
            for e in range(4):
                at = [(qd + 4 * e) * heads + col(qd + 4 * e, nt * 8 + g) for g in range(8) for qd in range(4)]
                assert len({a % 32 for a in at}) == 32
