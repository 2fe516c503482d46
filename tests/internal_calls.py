"""The library's internal launchers (csrc/common.h) for tests of single kernels:
its structs as ctypes, its launch functions by name."""
import ctypes as C
import os
import re
import subprocess

import paper_1606_06790_gb300 as pkg

CSRC = os.path.join(os.path.dirname(pkg.__file__), "csrc")
HEADER = open(os.path.join(CSRC, "common.h")).read()


def struct(name):
    body = re.search(r"struct %s \{(.*?)\n\};" % name, HEADER, re.S).group(1)
    fields = []
    for kind, names in re.findall(r"^\s*(int64_t|int|float|double) ([^;]+);", body, re.M):
        t = {"int64_t": C.c_int64, "int": C.c_int, "float": C.c_float, "double": C.c_double}[kind]
        for n in names.split(","):
            m = re.match(r"\s*(\w+)(?:\[(\d+)\])?\s*$", n)
            fields.append((m.group(1), t * int(m.group(2)) if m.group(2) else t))
    return type(name, (C.Structure,), {"_fields_": fields})


def launcher(name):
    lib = pkg.load_library()
    symbols = subprocess.run(["nm", "-D", lib._name], capture_output=True, text=True, check=True).stdout.split()
    return getattr(lib, next(s for s in symbols if re.match(r"_ZN5idmrg%d%s" % (len(name), name), s)))
