"""The forms of a helicity block agree (CPU; no GPU needed).

A block of g g -> t tbar g (g) takes a shorter form where the beams lie on the z axis; a
point turned off the axis, or with its beams along -z and +z, takes the general one, and
|M|^2 is the same.  The host build of the kernels' templates evaluates each point both ways,
with the colour sum of the blocks.

A turn rounds momenta at 1.1e-16 of the energy, an invariant s_ij at 1.1e-16 E^2 / s_ij; with
s_ij > 1e-3 E^2 (points are selected so) and some ten of them that is below 1e-11.  In float32
the invariants stay in float64 and products e.p and spinors round at 6e-8, over sqrt(s_ij) / E:
below 2e-5."""
import subprocess

import numpy as np
import pytest

import synth

PIDS = {"ee_uug": 1, "gg_ttg": 3, "gg_ttgg": 4, "uu_ttg": 6}


@pytest.fixture(scope="module")
def tool():
    from paper_2503_07439_gb300 import build
    try:
        return build.block_check_tool()
    except (RuntimeError, FileNotFoundError) as e:
        pytest.skip(f"CUDA toolchain unavailable: {e}")


def _blocks(tool, name, p):
    inp = f"{PIDS[name]} {p.shape[2]} {p.shape[1]}\n" + " ".join("%.17g" % x for x in p.reshape(-1)) + "\n"
    r = subprocess.run([tool], input=inp, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    v = np.array([[float(x) for x in line.split()] for line in r.stdout.split("\n") if line.strip()])
    return v[:, 0], v[:, 2]


def _points(name, n):
    p = synth.flat_points(name, 40 * n, 29).p
    ok = np.ones(p.shape[2], bool)
    for i in range(p.shape[1]):
        for j in range(i):
            s = p[0, i] * p[0, j] - (p[1:, i] * p[1:, j]).sum(0)
            ok &= 2 * s > 1e-3 * 4 * p[0, 0] ** 2
    assert ok.sum() >= n
    return np.ascontiguousarray(p[:, :, ok][:, :, :n])


def _turn(p, axis, angle):
    a = np.asarray(axis, float) / np.linalg.norm(axis)
    K = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    R = np.eye(3) + np.sin(angle) * K + (1 - np.cos(angle)) * K @ K
    q = p.copy()
    q[1:] = np.einsum("ab,bln->aln", R, p[1:])
    return q


@pytest.mark.parametrize("name", list(PIDS))
def test_block_forms_agree(tool, name):
    p = _points(name, 6 if name == "gg_ttgg" else 30)
    b64, b32 = _blocks(tool, name, p)
    flipped = p.copy()
    flipped[2:] *= -1.0  # half a turn about the x axis, exactly
    for q in (flipped, _turn(p, (1, 2, -1), 0.7), _turn(p, (0, 1, 0), 1e-9)):
        g64, g32 = _blocks(tool, name, q)
        assert np.max(np.abs(g64 / b64 - 1)) < 1e-11
        assert np.max(np.abs(g32 / b64 - 1)) < 2e-5
    assert np.max(np.abs(b32 / b64 - 1)) < 2e-5
