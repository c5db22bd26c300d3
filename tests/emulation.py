"""The decoder's library compiled for the host: the CUDA sources of csrc/ with their launches and inline PTX
statements rewritten, on the fibers of tests/host_emulation.  load() makes the Python package use it, with CPU tensors
in place of CUDA tensors and `STREAM` in place of a stream."""

import ctypes
import os
import re
import subprocess
import sys
import tempfile
import types

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_12262_gb300", "csrc")
HOST = os.path.join(ROOT, "tests", "host_emulation")
OUT = os.path.join(ROOT, "tests", "_build")
STREAM = types.SimpleNamespace(cuda_stream=0)


def _split(text):
    """Split at the commas outside brackets."""
    out, depth, cur = [], 0, ""
    for ch in text:
        depth += (ch in "([{") - (ch in ")]}")
        if ch == "," and depth == 0:
            out.append(cur.strip())
            cur = ""
        else:
            cur += ch
    return out + [cur.strip()] if cur.strip() else out


def _asm(match):
    code, operands = re.split(r"\s::?\s", match.group(1), maxsplit=1)
    code = "".join(re.findall(r'"((?:[^"\\]|\\.)*)"', code))
    args = [m.group(1) for m in (re.match(r'"=?[lr]"\s*(\(.*\))$', part, re.S)
                                 for part in _split(re.sub(r"\s:\s", ",", operands))) if m]
    if "globaltimer" in code:
        return "%s = emu::now_ns();" % args[0]
    if "st.release" in code:
        return "__atomic_store_n(%s, %s, __ATOMIC_RELEASE);" % tuple(args)
    if "cas.b128" in code:
        old0, old1, cmp0, cmp1, new0, new1, at = args
        return ("{ auto *q = (unsigned long long *)%s; %s = q[0]; %s = q[1]; if (q[0] == %s && q[1] == %s) "
                "{ q[0] = %s; q[1] = %s; } }" % (at, old0, old1, cmp0, cmp1, new0, new1))
    if "v2.b64" in code:
        return "{ auto *q = (const unsigned long long *)%s; %s = q[0]; %s = q[1]; }" % (args[2], args[0], args[1])
    if code.startswith("ld.relaxed.cta.b"):
        return "%s = *%s;" % tuple(args)
    raise ValueError("statement without a host counterpart: " + code)


def _translate(src):
    src = re.sub(r"asm volatile\((.*?)\);", _asm, src, flags=re.S)
    src = re.sub(r"extern __shared__ __align__\(16\) char (\w+)\[\];", r"char *\1 = emu::dynamic_shared();", src)
    return re.sub(r"(\w+(?:<[\w, ]*>)?)<<<(.*?)>>>\((.*?)\);",
                  lambda m: "emu::launch(%s, [&] { %s(%s); });" % (m.group(2), m.group(1), m.group(3)), src, flags=re.S)


def build(csrc=CSRC, out=None, flags=()):
    """Compile the sources of `csrc` (default: this repository's) and return the library's path."""
    out = out or OUT
    lib = os.path.join(out, "libqec_host.so")
    names = sorted(f for f in os.listdir(csrc) if f.endswith((".cu", ".cpp")))
    deps = [os.path.join(csrc, f) for f in os.listdir(csrc)] + [os.path.join(HOST, f) for f in os.listdir(HOST)] + \
        [os.path.abspath(__file__)]
    if os.path.exists(lib) and all(os.path.getmtime(d) < os.path.getmtime(lib) for d in deps):
        return lib
    os.makedirs(out, exist_ok=True)
    tag = ".%d" % os.getpid()
    jobs, objs, made = [], [], []
    for f in names + ["runtime.cpp"]:
        src = os.path.join(HOST if f == "runtime.cpp" else csrc, f)
        if f.endswith(".cu"):
            with open(src) as r:
                text = _translate(r.read())
            src = os.path.join(out, f + tag + ".cpp")
            with open(src, "w") as w:
                w.write(text)
            made.append(src)
        objs.append(os.path.join(out, f + tag + ".o"))
        cmd = ["g++", "-std=c++17", "-O1", "-fPIC", "-w", "-U_FORTIFY_SOURCE", "-I", HOST, "-I", csrc, *flags,
               "-c", src, "-o", objs[-1]]
        jobs.append((cmd, subprocess.Popen(cmd, stderr=subprocess.PIPE)))
    for cmd, p in jobs:
        err = p.communicate()[1]
        if p.returncode:
            raise RuntimeError(" ".join(cmd) + "\n" + err.decode(errors="replace")[:4000])
    subprocess.run(["g++", "-shared", "-o", lib + tag, *objs, *flags, "-lpthread"], check=True)
    os.replace(lib + tag, lib)
    for f in objs + made:
        os.remove(f)
    return lib


def program(code, source="decoder.cu", timeout=60):
    """Compile a C++ program around a translated source (its internal names are in reach) and run it."""
    lib = build()
    with open(os.path.join(CSRC, source)) as r:
        text = _translate(r.read())
    with tempfile.TemporaryDirectory() as tmp:
        src, exe = os.path.join(tmp, "program.cpp"), os.path.join(tmp, "program")
        with open(src, "w") as w:
            w.write(text + code)
        subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-U_FORTIFY_SOURCE", "-I", HOST, "-I", CSRC, src, lib,
                        "-Wl,-rpath," + os.path.dirname(lib), "-o", exe, "-lpthread"], check=True)
        return subprocess.run([exe], timeout=timeout, check=True, capture_output=True, text=True).stdout


def load(path=None, order=0, seed=1, sms=1):
    """The package on the host build; lanes run in order (0), in reverse (1) or at random (2)."""
    import paper_2609_12262_gb300 as q
    q.LIB_PATH = path or build()
    L = q.lib()
    L.emu_order.argtypes = [ctypes.c_int, ctypes.c_uint]
    L.emu_order(order, seed)
    L.emu_sms(sms)
    L.emu_barriers.restype = ctypes.c_longlong
    return q


def run(code, timeout=600):
    """Run Python code in a process of its own (an endless loop or an abort there is an exception here)."""
    build()
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, timeout=timeout, capture_output=True, text=True)
    if r.returncode:
        raise RuntimeError("exit %d\n%s\n%s" % (r.returncode, r.stdout[-2000:], r.stderr[-4000:]))
    return r.stdout
