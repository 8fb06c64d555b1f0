"""Variants of the library for tests, linked from the built objects: single
sources compiled with other macros, and host calls replaced by the linker."""
import os
import subprocess


def library(path, macros=None, wrap=(), source=""):
    """Links the library to `path`.  macros: {csrc file: [-D flags]}, compiled
    anew; wrap: functions whose calls go to __wrap_<name> in the C `source`
    (__real_<name> is the function itself).  Returns the loaded library, with
    its own state."""
    import paper_2202_05628_gb300 as art
    from paper_2202_05628_gb300 import build as b
    b.build()
    out = os.path.dirname(str(path))
    objs = []
    for cu in sorted(f for f in os.listdir(b.SRC) if f.endswith(".cu")):
        obj = os.path.join(b.OUT_DIR, cu[:-3] + ".o")
        if cu in (macros or {}):
            obj = os.path.join(out, cu[:-3] + ".o")
            subprocess.run([b.nvcc()] + b.ARCH + b.NVCC_FLAGS + macros[cu] + ["-c", os.path.join(b.SRC, cu), "-o", obj],
                           check=True)
        objs.append(obj)
    if source:
        c, obj = os.path.join(out, "wrap.c"), os.path.join(out, "wrap.o")
        with open(c, "w") as f:
            f.write(source)
        subprocess.run(["gcc", "-O1", "-fPIC", "-c", c, "-o", obj], check=True)
        objs.append(obj)
    flags = [x for w in wrap for x in ("-Xlinker", f"--wrap={w}")]
    subprocess.run([b.nvcc()] + b.ARCH + ["-shared", "-o", str(path)] + objs + flags + ["-lcuda"], check=True)
    return art.load_library(str(path))
