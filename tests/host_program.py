"""Small C++ programs over the library's own host code: compiled against its internal
headers and linked with its object files, for functions that need no GPU."""
import os
import subprocess


def build_program(directory, source):
    """Path of the program built from the C++ text `source` in `directory`."""
    from paper_2008_00326_gb300 import build
    build.build()
    objs = [os.path.join(build.BUILD_DIR, s.replace(".cu", ".o")) for s in build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    src, exe = os.path.join(str(directory), "program.cpp"), os.path.join(str(directory), "program")
    with open(src, "w") as f:
        f.write(source)
    subprocess.check_call([build._nvcc(), "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, src, *objs, "-o", exe])
    return exe
