"""The library built with other constants for a test: some of its units
compiled again with the given definitions, the others as they are."""
import concurrent.futures as cf
import os
import subprocess


def build_variant(out, units, definitions):
    """Path-like folder, names of units in csrc/, -D flags: the loaded library."""
    from paper_2203_02527_gb300 import _lib, build
    build.build()

    def compile_unit(name):
        subprocess.check_call([build._nvcc(), *build.NVCC_FLAGS, *definitions, "-c",
                               os.path.join(build.CSRC, name + ".cu"), "-o", str(out / (name + ".o"))])

    with cf.ThreadPoolExecutor(len(units)) as ex:
        list(ex.map(compile_unit, units))
    rest = [os.path.join(build.OUT_DIR, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    rest = [o for o in rest if os.path.basename(o)[:-2] not in units]
    lib = str(out / "libph0_variant.so")
    subprocess.check_call([build._nvcc(), *build.ARCH, "-shared", "-o", lib, *(str(out / (u + ".o")) for u in units),
                           *rest, "-lpthread"])
    return _lib.load(lib)
