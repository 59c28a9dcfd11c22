"""Builds the library's sources for the CPU emulation of cuda_runtime.h here.

The sources are taken as they are but for what a host compiler cannot parse:
launches, the few lines of PTX, dynamic shared memory, and the shared
variables that emu::Shared watches."""
import glob
import hashlib
import os
import re
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(os.path.dirname(HERE))
CSRC = os.path.join(ROOT, "paper_2203_02228_gb300", "csrc")
LEFT_OUT = ("probe.cu",)                # a bandwidth probe: PTX throughout
NOT_WATCHED = ("s_cur", "s_mv", "s_pmv", "mv")  # polled on purpose; passed on as plain pointers
WATCHED_STRUCTS = ("KnnBuf", "LsShared", "FbBlock")


def _launch(m):
    name, cfg, args = m.groups()
    parts, depth = [""], 0
    for ch in cfg:
        depth += (ch in "([") - (ch in ")]")
        if ch == "," and depth == 0:
            parts.append("")
        else:
            parts[-1] += ch
    smem = parts[2] if len(parts) > 2 else "0"
    return "emu::launch(dim3(%s), dim3(%s), %s, [=] { %s(%s); });" % (parts[0], parts[1], smem, name, args)


def _watch(m):
    decl = m.group(0)
    names = re.findall(r"(\w+)(?:\[[^\]]*\])*\s*[,;]", decl)
    if any(n in NOT_WATCHED for n in names):
        return decl
    return re.sub(r"\b(int|int32_t|int64_t|uint64_t|int2)\b", r"emu::Shared<\1>", decl, count=1)


def _host_source(s):
    s = s.replace("__noinline__", "")  # (a macro of that name would break the C++ library's headers)
    s = re.sub(r"extern __shared__\s+(?:__align__\(16\)\s+)?(\w+)\s+(\w+)\[\];",
               r"\1* \2 = reinterpret_cast<\1*>(emu::dyn);", s)
    s = re.sub(r"__shared__ (?:int|int32_t|int64_t|int2) [^;]*;", _watch, s)
    for name in WATCHED_STRUCTS:
        s = re.sub(r"struct %s \{.*?\n\};" % name,
                   lambda m: re.sub(r"^  \w+ [^;/]*;", _watch, m.group(0), flags=re.M), s, flags=re.S)
    s = s.replace("redo_list[atomicAdd(redo_n, 1)] = e", "emu::append_once(redo_list, redo_n, e)")
    s = re.sub(r'asm volatile\("mov.u64 %0, %%globaltimer;"[^;]*;', "static uint64_t ns; t = ++ns;", s)
    s = re.sub(r'asm\("sqrt[^"]*"[^;]*;', "r = sqrtf(x);", s)
    s = re.sub(r'asm volatile\("prefetch[^"]*"[^;]*;', ";", s)
    return re.sub(r"([A-Za-z_]\w*(?:<[\w, ]+>)?)<<<(.*?)>>>\((.*?)\);", _launch, s, flags=re.S)


def build():
    """Path of the emulated library (kept under _build/ by what went into it)."""
    files = sorted(glob.glob(os.path.join(CSRC, "*"))) + sorted(glob.glob(os.path.join(HERE, "*.*")))
    files += sorted(glob.glob(os.path.join(ROOT, "include", "*.h")))
    h = hashlib.sha256()
    for f in files:
        with open(f, "rb") as fh:
            h.update(fh.read())
    out = os.path.join(HERE, "_build", h.hexdigest()[:16])
    lib = os.path.join(out, "libfaco_emu.so")
    if os.path.exists(lib):
        return lib
    os.makedirs(out, exist_ok=True)
    for f in files:
        if os.path.dirname(f) == CSRC and f.endswith((".cu", ".cuh", ".h", ".inc")):
            with open(f) as fh, open(os.path.join(out, os.path.basename(f)), "w") as to:
                to.write(_host_source(fh.read()))
    with open(os.path.join(out, "probe.cpp"), "w") as to:
        to.write('extern "C" int faco_l2_probe(unsigned long, int, double*) { return -4; }\n')
    units = [f for f in glob.glob(os.path.join(out, "*.cu")) if os.path.basename(f) not in LEFT_OUT]
    units += [os.path.join(out, "probe.cpp"), os.path.join(HERE, "emu.cpp")]
    objs = [os.path.join(out, os.path.basename(u) + ".o") for u in units]
    flags = ["-std=c++17", "-O1", "-fPIC", "-w", "-ffp-contract=off", "-U_FORTIFY_SOURCE",
             "-I", HERE, "-I", out, "-I", os.path.join(ROOT, "include")]
    with ThreadPoolExecutor(8) as ex:
        done = list(ex.map(lambda uo: subprocess.run(["g++", "-x", "c++"] + flags + ["-c", uo[0], "-o", uo[1]],
                                                     capture_output=True, text=True), zip(units, objs)))
    for d in done:
        if d.returncode:
            sys.stderr.write(d.stderr)
            raise RuntimeError("the emulated library does not compile")
    tmp = "%s.%d" % (lib, os.getpid())
    subprocess.run(["g++", "-shared", "-o", tmp] + objs + ["-lpthread"], check=True)
    for o in objs:
        os.remove(o)
    os.replace(tmp, lib)
    return lib
