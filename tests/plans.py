"""The kernel entry that a call takes (tests/plan_probe.cpp, linked with the library's objects):
the tests that name an entry, or stand at the edge of one, check here that they do."""
import os
import subprocess

from paper_2609_37241_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
_exe = None


def _probe():
    global _exe
    if _exe is None:
        build.build()
        src, exe = os.path.join(HERE, "plan_probe.cpp"), os.path.join(build.BUILD, "plan_probe")
        objs = [os.path.join(build.BUILD, s + ".o") for s in build.SOURCES]
        deps = objs + [src, os.path.join(build.CSRC, "internal.h")]
        if not os.path.exists(exe) or any(os.path.getmtime(d) > os.path.getmtime(exe) for d in deps):
            subprocess.run([build.nvcc(), "-std=c++17", "-I", build.CSRC, "-I", build.INC, src, *objs,
                            "-o", exe + ".tmp"], check=True)
            os.replace(exe + ".tmp", exe)
        _exe = exe
    return _exe


def plans(lines):
    out = subprocess.run([_probe()], input="".join(ln + "\n" for ln in lines), capture_output=True, text=True,
                         check=True).stdout.splitlines()
    assert len(out) == len(lines)
    return out


def norm(res, dtype, H, T, off=0, rs=None):
    return plans([f"norm {int(res)} {dtype} {H} {T} {off} {H if rs is None else rs}"])[0]


def rope(T, Hq, Hkv, D, qk, any_align=False):
    return plans([f"rope {int(any_align)} {int(qk)} {Hq} {Hkv} {D} {T}"])[0]


# Norm calls at the limits of their entries: (dtype, T, H, rows' element offset from a 16-byte boundary,
# entry with the residual, entry without); BF16 1, FP16 2, FP32 3.
NORM_LIMITS = [
    (1, 608, 6144, 0, "vec", "vec"), (1, 609, 6144, 0, "large_bulk", "large_bulk"),     # two waves of blocks
    (2, 152, 12296, 0, "vec", "vec"), (1, 153, 12288, 0, "large_bulk", "large_bulk"),   # one, two vectors each
    (1, 1217, 2048, 0, "mid", "vec"), (2, 690, 4096, 0, "mid", "mid"), (1, 608, 4096, 0, "vec", "vec"),
    (2, 1217, 4096, 0, "large_regs", "large_bulk"), (1, 609, 8192, 0, "mid", "large_bulk"),
    (2, 913, 8192, 0, "large_bulk", "large_bulk"),
    (3, 1217, 2048, 0, "vec", "large_regs"), (3, 457, 5000, 0, "vec", "large_regs"),    # four per thread
    (3, 305, 8192, 0, "vec", "large_regs"), (3, 305, 7000, 0, "vec", "large_regs"),     # eight
    (1, 1368, 264, 0, "few", "few"), (1, 1369, 264, 0, "vec", "vec"),  # few rows
    (2, 2128, 1024, 0, "few", "few"), (2, 2129, 1024, 0, "few", "vec"), (3, 6081, 512, 0, "vec", "vec"),
    (3, 1, 148, 0, "few", "few"), (1, 152, 16384, 0, "few", "few"), (2, 153, 16384, 0, "large_bulk", "large_bulk"),
    (3, 61, 8192, 0, "few", "few"), (3, 77, 8192, 0, "few", "vec"), (3, 60, 8192, 0, "vec", "few"),
    (1, 475, 333, 1, "edge", "edge"), (2, 713, 333, 1, "edge_flat", "edge_flat"),       # rows at odd offsets
    (1, 1354, 333, 1, "edge", "edge_flat"), (2, 357, 1023, 1, "edge_flat", "edge_flat"),
    (1, 88, 4001, 1, "edge_flat", "edge"), (2, 91, 4095, 1, "edge_flat", "edge_flat"),
    (1, 40, 9001, 1, "edge", "edge"), (2, 85, 9007, 1, "edge_flat", "edge_flat"),       # two vectors per thread
]

# RoPE calls at the limits of their entries: (T, Hq, Hkv, D, q/k norm, entry and block size).
ROPE_LIMITS = [
    (38, 32, 8, 128, False, "one_64"), (39, 32, 8, 128, False, "two_64"), (115, 32, 8, 128, False, "two_64"),
    (116, 32, 8, 128, False, "one_256"), (139, 32, 8, 128, False, "one_128"), (152, 32, 8, 128, False, "one_128"),
    (153, 32, 8, 128, False, "one_256"), (304, 32, 8, 128, False, "one_256"), (305, 32, 8, 128, False, "two_64"),
    (575, 32, 8, 128, False, "two_64"), (576, 32, 8, 128, False, "bulk_128"),
    (57, 32, 8, 128, True, "one_64"), (58, 32, 8, 128, True, "two_64"), (87, 32, 8, 128, True, "two_64"),
    (88, 32, 8, 128, True, "one_128"), (405, 32, 8, 128, True, "one_128"), (406, 32, 8, 128, True, "two_64"),
    (347, 16, 4, 64, False, "one_64"), (405, 16, 4, 64, False, "one_64"), (406, 16, 4, 64, False, "one_256"),
    (511, 5, 1, 128, True, "two_64"), (400, 3, 2, 256, False, "one_256"), (333, 3, 3, 256, True, "one_128"),
]
