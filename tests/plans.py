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


def chain(qk, H, Hq, I, T, pdl=True, inplace=False, Hkv=8):
    return plans([f"chain {int(qk)} {H} {Hq} {Hkv} {I} {T} {int(inplace)} {int(pdl)}"])[0]


# Norm calls at the limits of their entries: (dtype, T, H, rows' element offset from a 16-byte boundary,
# entry with the residual, entry without); BF16 1, FP16 2, FP32 3.
NORM_LIMITS = [
    (1, 608, 6144, 0, "vec", "vec"), (1, 609, 6144, 0, "large_bulk", "large_bulk"),     # two waves of blocks
    (2, 152, 12296, 0, "vec", "vec"), (1, 153, 12288, 0, "large_bulk", "large_bulk"),   # one, two vectors each
    (2, 311, 8448, 0, "large_bulk", "large_bulk"), (1, 157, 12288, 0, "large_bulk", "large_bulk"),
    (2, 160, 12296, 0, "large_bulk", "large_bulk"), (1, 161, 16384, 0, "large_bulk", "large_bulk"),
    (1, 1217, 2048, 0, "mid", "vec"), (2, 690, 4096, 0, "mid", "mid"), (1, 608, 4096, 0, "vec", "vec"),
    (2, 1217, 4096, 0, "large_regs", "large_bulk"), (1, 609, 8192, 0, "mid", "large_bulk"),
    (2, 913, 8192, 0, "large_bulk", "large_bulk"),
    (3, 1217, 2048, 0, "vec", "large_regs"), (3, 457, 5000, 0, "vec", "large_regs"),    # four per thread
    (3, 305, 8192, 0, "vec", "large_regs"), (3, 305, 7000, 0, "vec", "large_regs"),     # eight
    (1, 1368, 264, 0, "few", "few"), (1, 1369, 264, 0, "vec", "vec"),  # few rows
    (2, 2128, 1024, 0, "few", "few"), (2, 2129, 1024, 0, "few", "vec"), (2, 2432, 1024, 0, "few", "vec"), (3, 2433, 512, 0, "vec", "vec"),
    (3, 1, 148, 0, "few", "few"), (1, 152, 16384, 0, "few", "few"), (2, 153, 16384, 0, "large_bulk", "large_bulk"),
    (3, 61, 8192, 0, "few", "few"), (3, 77, 8192, 0, "few", "vec"), (3, 60, 8192, 0, "vec", "few"),
    (1, 475, 333, 1, "edge", "edge"), (2, 713, 333, 1, "edge_flat", "edge_flat"),       # rows at odd offsets
    (1, 1354, 333, 1, "edge", "edge_flat"), (2, 357, 1023, 1, "edge_flat", "edge_flat"),
    (1, 88, 4001, 1, "edge_flat", "edge"), (2, 91, 4095, 1, "edge_flat", "edge_flat"),
    (2, 304, 9501, 1, "edge", "edge"), (2, 305, 9501, 1, "edge", "edge_many"),     # more per thread
    (1, 305, 10241, 1, "edge", "edge_many"), (1, 306, 12287, 1, "edge", "edge_many"),
    (1, 3799, 12299, 1, "edge", "edge"), (2, 3801, 12301, 1, "edge", "edge_many"),      # scalar accesses
    (3, 152, 5601, 1, "edge", "edge"), (3, 153, 5601, 1, "edge", "edge_many"), (3, 157, 8191, 1, "edge", "edge_many"),
    (3, 912, 4501, 1, "edge", "edge"), (3, 913, 4501, 1, "edge", "edge_many"),
    (3, 1023, 2222, 1, "edge", "edge"), (3, 1025, 2222, 1, "edge", "edge_many"),
    (1, 40, 9001, 1, "edge", "edge"), (2, 85, 9007, 1, "edge", "edge"),                 # two vectors per thread
]

# RoPE calls at the limits of their entries: (T, Hq, Hkv, D, q/k norm, entry and block size).
ROPE_LIMITS = [
    (38, 32, 8, 128, False, "one_64"), (39, 32, 8, 128, False, "two_64"), (133, 32, 8, 128, False, "two_64"),
    (134, 32, 8, 128, False, "one_64"), (153, 32, 8, 128, False, "two_64"), (190, 32, 8, 128, False, "one_64"),
    (191, 32, 8, 128, False, "two_64"), (575, 32, 8, 128, False, "two_64"), (576, 32, 8, 128, False, "bulk_128"),
    (57, 32, 8, 128, True, "one_64"), (58, 32, 8, 128, True, "two_64"), (76, 32, 8, 128, True, "two_64"),
    (77, 32, 8, 128, True, "one_64"), (342, 32, 8, 128, True, "one_64"), (343, 32, 8, 128, True, "two_64"),
    (511, 5, 1, 128, True, "one_64"), (400, 3, 2, 256, False, "one_64"), (333, 3, 3, 256, True, "one_64"),
    (230, 32, 8, 64, False, "two_64"), (231, 32, 8, 64, False, "one_256"), (280, 32, 8, 64, False, "one_128"),
    (305, 32, 8, 64, False, "one_256"), (608, 32, 8, 64, False, "one_256"), (609, 32, 8, 64, False, "two_64"),
    (347, 16, 4, 64, False, "one_64"), (406, 16, 4, 64, False, "one_256"), (1152, 32, 8, 64, False, "bulk_128"),
    (114, 32, 8, 64, True, "one_64"), (115, 32, 8, 64, True, "two_64"), (174, 32, 8, 64, True, "two_64"),
    (175, 32, 8, 64, True, "one_128"), (810, 32, 8, 64, True, "one_128"), (811, 32, 8, 64, True, "two_64"),
]

# Layer-chain calls at the limits of their entries: (H, q heads, I, q/k norm, T, PDL, in place, plan);
# 8 k/v heads of D 128. The plan: norm CTAs per token (two, one, or one with wide SwiGLU tiles), late
# trigger, token-major order; head-rows per RoPE lane group, items per RoPE block.
CHAIN_LIMITS = [
    (4096, 32, 14336, False, 4, True, False, "two_tok rows1 ipb4"), (4096, 32, 14336, False, 5, True, False, "two_late rows1 ipb4"),
    (4096, 32, 14336, False, 13, True, False, "two_late rows1 ipb8"), (4096, 32, 14336, False, 72, True, False, "two_late rows1 ipb8"),
    (4096, 32, 14336, False, 73, True, False, "two rows1 ipb8"), (4096, 32, 14336, False, 81, True, False, "two rows1 ipb8"),
    (4096, 32, 14336, False, 82, True, False, "one_late rows1 ipb8"), (4096, 32, 14336, False, 94, True, False, "one_late rows3 ipb8"),
    (4096, 32, 14336, False, 116, True, False, "one_late rows3 ipb8"), (4096, 32, 14336, False, 117, True, False, "one rows3 ipb8"),
    (4096, 32, 14336, False, 40, False, False, "two_tok rows1 ipb8"), (4096, 32, 14336, False, 41, False, False, "two rows1 ipb8"),
    (4096, 32, 14336, False, 82, False, False, "one rows1 ipb8"),
    (4096, 32, 12288, True, 30, True, False, "two_late rows1 ipb4"), (4096, 32, 12288, True, 31, True, False, "two_late rows1 ipb8"),
    (4096, 32, 12288, True, 100, True, False, "one_late rows1 ipb8"), (4096, 32, 12288, True, 117, True, False, "one rows1 ipb8"),
    (4096, 32, 12288, True, 139, True, False, "one rows3 ipb8"),
    (8192, 64, 28672, False, 1, True, False, "two_tok rows1 ipb4"), (8192, 64, 28672, False, 10, True, False, "two_late rows1 ipb4"),
    (8192, 64, 28672, False, 11, True, False, "two_late rows1 ipb8"), (8192, 64, 28672, False, 28, True, False, "two rows1 ipb16"),
    (8192, 64, 28672, False, 31, True, False, "one_late rows1 ipb16"), (8192, 64, 28672, False, 33, True, False, "wide_late rows1 ipb16"),
    (8192, 64, 28672, False, 49, True, False, "wide_late rows3 ipb16"), (8192, 64, 28672, False, 56, True, False, "wide rows3 ipb16"),
    (8192, 64, 28672, True, 25, True, False, "two_late rows1 ipb8"), (8192, 64, 28672, True, 26, True, False, "two_late rows1 ipb16"),
    (8192, 64, 28672, True, 48, True, False, "wide_late rows1 ipb16"), (8192, 64, 28672, True, 49, True, False, "wide rows1 ipb16"),
    (8192, 64, 28672, True, 83, True, False, "wide rows3 ipb16"),
    (4096, 32, 14336, False, 4, True, True, "one_tok rows1 ipb4"), (4096, 32, 14336, False, 14, True, True, "one_late rows1 ipb4"),
    (4096, 32, 14336, False, 100, True, True, "one_late rows3 ipb8"), (4096, 32, 14336, False, 130, True, True, "one rows3 ipb8"),
    (8192, 64, 22016, True, 12, True, True, "one_late rows1 ipb4"), (8192, 64, 22016, True, 50, True, True, "wide_late rows1 ipb16"),
    (8192, 64, 22016, True, 60, True, True, "wide rows1 ipb16"), (8192, 64, 22016, True, 100, True, True, "wide rows3 ipb16"),
]
