"""The selection minor loop's device code on the CPU under ThreadSanitizer
(select_emulator.cpp): no unordered accesses to shared or global memory, no
barrier that part of a block misses, and the oracle's bits."""
import os
import re
import subprocess

import numpy as np
import pytest

import oracle
import paper_2501_01461_gb300 as cg
import synth

HERE = os.path.dirname(os.path.abspath(__file__))
PKG = os.path.dirname(cg.__file__)
FLAGS = ["-std=c++17", "-O1", "-g", "-ffp-contract=off", "-frounding-math", "-pthread", "-w",
         "-I" + os.path.join(PKG, "csrc"), "-I" + os.path.join(os.path.dirname(HERE), "include"),
         "-I/usr/local/cuda/include", "-fsanitize=thread"]


def _spell_out(m):
    """An inline PTX load or store as C."""
    op, args = m.group(1), re.findall(r'"(=?\w)"\(([^)]*)\)', m.group(2))
    outs, ins = [a for a in args if a[0][0] == "="], [a for a in args if a[0][0] != "="]
    p = ins[0][1]
    if op.startswith("ld.acquire"):
        return f"{outs[0][1]} = __atomic_load_n({p}, __ATOMIC_ACQUIRE);"
    if op.startswith("st.release"):
        return f"__atomic_store_n({p}, {ins[1][1]}, __ATOMIC_RELEASE);"
    assert op.startswith("ld.global") and all(o[0] == "=f" for o in outs), op
    return " ".join(f"{o} = ((const float*)({p}))[{i}];" for i, (_, o) in enumerate(outs))


def device_code(threads):
    """minor_select.cu without its launches, with blocks of `threads`."""
    src = open(os.path.join(PKG, "csrc", "minor_select.cu")).read()
    src = src[:src.index("cudaError_t select_build_psf")] + "}  // namespace cleangb\n"
    src = re.sub(r'#include "[^"]*"', "", src)
    src = re.sub(r'asm volatile\(\s*"(\S+) [^"]*"\s*(.*?)\);', _spell_out, src, flags=re.S)
    src = re.sub(r"\*\(volatile ([\w ]+)\*\)(&?[\w>.\-]+(\[[^\]]*\])?)",
                 r"relaxed_load((\1*)(\2))", src)
    assert "volatile" not in re.sub(r"//.*", "", src)
    src, n = re.subn(r"extern __shared__[^;]*;", "", src)
    assert n == 1
    src, n = re.subn(r"constexpr int kThreads = \d+;", f"constexpr int kThreads = {threads};", src)
    assert n == 1 and "asm" not in re.sub(r"//.*", "", src)
    return src


_built = {}


@pytest.fixture(scope="module")
def emulator(tmp_path_factory):
    def build(threads):
        if threads not in _built:
            d = tmp_path_factory.mktemp(f"emu{threads}")
            (d / "select_device.inc").write_text(device_code(threads))
            exe = str(d / "emu")
            r = subprocess.run(["g++", *FLAGS, f"-I{d}", os.path.join(HERE, "select_emulator.cpp"),
                                "-o", exe], capture_output=True, text=True)
            if r.returncode != 0 and ("sanitize" in r.stderr or "tsan" in r.stderr):
                pytest.skip("ThreadSanitizer unavailable")
            assert r.returncode == 0, r.stderr[-4000:]
            _built[threads] = exe
        return _built[threads]
    return build


def _emulate(exe, tmp_path, dirty, psf, gain, niter, thr, tiles, G, plain_cycles=0.0, force=0):
    """(residual, model, components, tiles' hand-over keys) of one launch; None
    for one whose waits were made to expire and did."""
    ny, nx = dirty.shape
    inp, out = tmp_path / "in", tmp_path / "out"
    inp.write_bytes(np.array([ny, nx, *psf.shape, *tiles, G, force], np.int32).tobytes()
                    + np.int64(niter).tobytes() + np.array([gain, thr, plain_cycles], np.float32).tobytes()
                    + dirty.tobytes() + psf.tobytes())
    r = subprocess.run([exe, str(inp), str(out)], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, TSAN_OPTIONS="halt_on_error=0 exitcode=66"))
    if "unexpected memory mapping" in r.stderr:
        pytest.skip("ThreadSanitizer cannot run here")
    if force and r.returncode == 5:
        return None
    assert r.returncode == 0, (r.returncode, r.stderr[:3000])
    b = out.read_bytes()
    n = ny * nx
    f = np.frombuffer(b, np.float32, 2 * n)
    comps, keys, at = [], [], 8 * n
    for _ in range(tiles[0] * tiles[1]):
        k = int(np.frombuffer(b, np.int32, 1, at)[0])
        keys.append(int(np.frombuffer(b, np.uint64, 1, at + 4)[0]))
        comps.append(np.frombuffer(b, cg.COMPONENT_DTYPE, k, at + 12))
        at += 12 + 16 * k
    return f[:n].reshape(ny, nx), f[n:].reshape(ny, nx), np.concatenate(comps), keys


def _field(ny, nx, ps, seed):
    rng = np.random.default_rng(seed)
    big = synth.make_psf(2 * ps[0], 2 * ps[1])
    psf = np.ascontiguousarray(big[ps[0] - ps[0] // 2:, ps[1] - ps[1] // 2:][:ps[0], :ps[1]])
    dirty = synth.random_image(ny, nx, rng, 1e-3)
    for _ in range(4):
        y, x = rng.integers(ny), rng.integers(nx)
        y0, x0 = max(0, y - ps[0] // 2), max(0, x - ps[1] // 2)
        sub = psf[y0 - y + ps[0] // 2:, x0 - x + ps[1] // 2:][:ny - y0, :nx - x0]
        dirty[y0:y0 + sub.shape[0], x0:x0 + sub.shape[1]] += np.float32(rng.uniform(0.1, 2)) * sub
    return dirty, psf


def _check(emulator, tmp_path, dirty, psf, niter, thr=0.0, tiles=(1, 1), G=1, threads=64,
           gain=0.1):
    o = oracle.clean_f32(dirty, psf, gain, niter, thr, tiles, 0)
    r, m, c, keys = _emulate(emulator(threads), tmp_path, dirty, psf, gain, niter, thr, tiles, G)
    assert not any(keys)
    for k in ("y", "x", "tile"):
        assert np.array_equal(c[k], o.comps[k]), (k, c[k], o.comps[k])
    assert np.array_equal(c["flux"].view(np.uint32), o.comps["flux"].view(np.uint32))
    assert np.array_equal(r.view(np.uint32), o.residual.view(np.uint32))
    assert np.array_equal(m.view(np.uint32), o.model.view(np.uint32))


def test_first_candidates(emulator, tmp_path):
    """A selection of two components: the candidates' first threshold is kept,
    which every thread of the block decides from one shared count."""
    dirty, psf = _field(64, 64, (128, 128), 64)
    dirty[10, 50], dirty[50, 10] = 3.0, 2.9
    _check(emulator, tmp_path, dirty, psf, 2)


@pytest.mark.parametrize("ny,nx,ps,niter,G,threads", [
    (64, 64, (128, 128), 90, 1, 64),     # cells kept singly; more than one selection
    (61, 45, (61, 45), 30, 2, 64),       # a group of two, a clipped PSF, ragged cells
    (40, 56, (81, 113), 70, 3, 128),
    (16, 17000, (32, 34000), 70, 2, 256),  # superblocks
])
def test_no_races_and_the_oracles_bits(emulator, tmp_path, ny, nx, ps, niter, G, threads):
    dirty, psf = _field(ny, nx, ps, ny)
    _check(emulator, tmp_path, dirty, psf, niter, G=G, threads=threads)


def test_more_ties_than_candidates(emulator, tmp_path):
    """One component a selection: it ends before its first barrier between
    reading the tile's margin and writing it."""
    psf = np.zeros((200, 220), np.float32)
    psf[100, 110] = 1.0
    dirty = synth.tie_image(100, 110, np.random.default_rng(3))
    _check(emulator, tmp_path, dirty, psf, 20, tiles=(1, 2), gain=0.5)


def test_resolved_cells_that_add_candidates(emulator, tmp_path):
    rng = np.random.default_rng(5)
    _check(emulator, tmp_path, synth.random_image(64, 48, rng), synth.random_psf(60, 50, rng), 150)


def test_cells_with_nan_pixels(emulator, tmp_path):
    """A PSF that makes the residual overflow, and no wider than 3 pixels: some
    pixels of a cell turn NaN, and its others still rise to the peak."""
    dirty = synth.random_image(64, 64, np.random.default_rng(1), 1e-2)
    dirty[10, 62], dirty[13, 61] = 3e38, 5.0
    psf = np.zeros((3, 3), np.float32)
    psf[1, 1] = psf[1, 2] = 400.0
    _check(emulator, tmp_path, dirty, psf, 12)


@pytest.mark.parametrize("G", [1, 2])
def test_tile_handed_over_to_the_plain_loop(emulator, tmp_path, G):
    """Against a plain loop that costs nothing every selection is slow: after
    two the round stops, the residual holds every component, and the key is
    that of its peak."""
    dirty, psf = _field(48, 40, (96, 80), 3)
    r, m, c, (key,) = _emulate(emulator(64), tmp_path, dirty, psf, 0.1, 300, 0.0, (1, 1), G, 1e-6)
    assert 2 <= len(c) <= 128
    o = oracle.clean_f32(dirty, psf, 0.1, len(c), 0.0, (1, 1), 0)
    assert np.array_equal(c["y"], o.comps["y"]) and np.array_equal(c["x"], o.comps["x"])
    assert np.array_equal(r.view(np.uint32), o.residual.view(np.uint32))
    assert np.array_equal(m.view(np.uint32), o.model.view(np.uint32))
    i = int(np.abs(r).argmax())
    v = int(r.ravel()[i].view(np.uint32))
    assert key == ((v & 0x7fffffff) << 32 | (0x7fffffff - i) << 1 | v >> 31)


def test_waits_of_a_group_that_expire(emulator, tmp_path):
    """Rank 0 waits for an arrival that never comes, the others for its post: all
    return in bounded time, the launch reports it, and no tile is handed over."""
    dirty, psf = _field(48, 40, (96, 80), 3)
    for plain_cycles in (0.0, 1e-6):
        assert _emulate(emulator(64), tmp_path, dirty, psf, 0.1, 300, 0.0, (1, 1), 3,
                        plain_cycles, force=1) is None
