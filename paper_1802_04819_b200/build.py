"""Compile the CUDA library in-tree with nvcc for sm_100a."""

from __future__ import annotations

import subprocess
import sysconfig
import tempfile
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
CSRC = PKG / "csrc"
LIB = PKG / "libslaq.so"
MARSHAL = PKG / "_marshal.so"      # Python extension: argument marshalling of the loop's two calls
SOURCES = ["slaq_api.cu", "slaq_fit.cu", "slaq_gain.cu", "slaq_alloc.cu", "slaq_select.cu", "slaq_pipe.cu"]


# Instrumented builds of the same sources, each a library of its own beside libslaq.so.
VARIANTS = {
    "clocks": ["-DSLAQ_PHASE_CLOCKS"],     # the fit kernel times its phases (slaq_get_fit_phase_cycles)
    "bounds": ["-DSLAQ_DEBUG_BOUNDS"],     # every ring, pool, gain, segment and shared-slice index is checked
}


def variant_path(name: str) -> Path:
    return PKG / f"libslaq_{name}.so"


def compile_library(out: Path = LIB, defines=(), verbose_ptxas: bool = False) -> None:
    """One nvcc per source, side by side, and a link: the fit's kernels alone take as long as everything else together.
    Device code is not compressed: unpacking it took 11 of the 26 ms of a process's first handle."""
    arch = ["nvcc", "-gencode", "arch=compute_100a,code=sm_100a"]
    flags = ["-lineinfo", "-O3", "--compress-mode=none", "-std=c++17", "-I", str(ROOT / "include"), "-Xcompiler", "-fPIC", *defines]
    if verbose_ptxas:
        flags += ["-Xptxas", "-v"]
    with tempfile.TemporaryDirectory() as tmp:
        objects = [str(Path(tmp) / (Path(s).stem + ".o")) for s in SOURCES]
        running = [subprocess.Popen([*arch, *flags, "-c", "-o", o, str(CSRC / s)]) for s, o in zip(SOURCES, objects)]
        failed = [s for s, p in zip(SOURCES, running) if p.wait()]
        if failed:
            raise RuntimeError(f"nvcc failed on {', '.join(failed)}")
        subprocess.run([*arch, "-Xcompiler", "-fPIC", "-shared", "-o", str(out), *objects], check=True)


def build_variant(name: str, force: bool = False) -> Path:
    """Compile an instrumented build (see VARIANTS) to libslaq_<name>.so."""
    out = variant_path(name)
    if force or is_stale(out):
        compile_library(out, VARIANTS[name])
    return out


def is_stale(lib: Path = LIB) -> bool:
    if not lib.exists():
        return True
    built = lib.stat().st_mtime
    deps = list(CSRC.glob("*.cu")) + list(CSRC.glob("*.cuh")) + [ROOT / "include" / "slaq.h"]
    return any(d.stat().st_mtime > built for d in deps)


def build_marshal(force: bool = False) -> Path:
    source = CSRC / "marshal.c"
    if force or not MARSHAL.exists() or source.stat().st_mtime > MARSHAL.stat().st_mtime:
        subprocess.run(["gcc", "-O2", "-Wall", "-Wextra", "-fPIC", "-shared", "-I", sysconfig.get_paths()["include"],
                        "-o", str(MARSHAL), str(source)], check=True)
    return MARSHAL


def build(force: bool = False, verbose_ptxas: bool = False) -> Path:
    build_marshal(force)
    if force or verbose_ptxas or is_stale():
        compile_library(verbose_ptxas=verbose_ptxas)
    return LIB


if __name__ == "__main__":
    build(force=True, verbose_ptxas=True)
