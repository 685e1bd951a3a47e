"""What the kernels evaluate, on the host (CPU; no GPU needed).

csrc/me_blockcheck.cu compiles the kernels' own block sums and closed forms for the host:
the closed helicity blocks of e+e- -> u ubar g, the 2 -> 2 trees, and the blocks with the colour
sum of the kernels.  They are compared with the helicities taken one at a time, and with
themselves at other scales of the momenta.

Scale: |M|^2 has the dimension E^(2 (4 - n_ext)), so momenta and masses scaled by a power of
two give the same value scaled by a power of two, exactly, as long as no intermediate leaves
the range of the arithmetic."""
import subprocess

import numpy as np
import pytest

import synth

PIDS = {"ee_uu": 0, "ee_uug": 1, "gg_tt": 2, "gg_ttg": 3, "gg_ttgg": 4, "uu_tt": 5, "uu_ttg": 6}


@pytest.fixture(scope="module")
def tool():
    from paper_2503_07439_gb300 import build
    try:
        return build.block_check_tool()
    except (RuntimeError, FileNotFoundError) as e:
        pytest.skip(f"CUDA toolchain unavailable: {e}")


def _run(tool, name, p, *args):
    inp = f"{PIDS[name]} {p.shape[2]} {p.shape[1]}\n" + " ".join("%.17g" % x for x in p.reshape(-1)) + "\n"
    r = subprocess.run([tool, *map(str, args)], input=inp, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    return np.array([[float(x) for x in line.split()] for line in r.stdout.split("\n") if line.strip()]).T


def _points(name, n):
    """Flat points whose invariants are above a thousandth of s (less with six legs)."""
    p = synth.flat_points(name, 40 * n, 31).p
    s = np.min([p[0, i] * p[0, j] - (p[1:, i] * p[1:, j]).sum(0) for i in range(p.shape[1]) for j in range(i)], axis=0)
    p = p[:, :, 2 * s > (4e-4 if name == "gg_ttgg" else 1e-3) * 4 * p[0, 0] ** 2]
    assert p.shape[2] >= n
    return np.ascontiguousarray(p[:, :, :n])


@pytest.mark.parametrize("name", list(PIDS))
def test_kernel_values_equal_single_helicities(tool, name):
    """Float64 rounds an invariant s_ij at 1.1e-16 s / s_ij, below 1e-12 with some ten of them;
    float32 values, from invariants in float64, are within 2e-6 of it."""
    p = _points(name, 4 if name == "gg_ttgg" else 30)
    _, s64, _, _ = _run(tool, name, p)
    v64, v32 = _run(tool, name, p, "kernels", 173.0)
    assert np.max(np.abs(v64 / s64 - 1)) < 1e-12
    assert np.max(np.abs(v32 / s64 - 1)) < (2e-5 if name == "gg_ttgg" else 2e-6)


# The powers of two up to which float32 evaluates these points (100 GeV with e+e-, 1 TeV, 2 TeV with
# six legs) without leaving its range 2^-126 .. 2^127.  Where |M|^2 falls like E^0, E^-2 and E^-4
# with 4, 5 and 6 legs, the ends come from single reciprocal invariants, of order E^-2, and, with
# colour flows, from squares of amplitudes.
RANGE = {"ee_uu": (-50, 50), "ee_uug": (-50, 50), "gg_tt": (-50, 50), "gg_ttg": (-48, 34), "gg_ttgg": (-34, 23),
         "uu_tt": (-50, 50), "uu_ttg": (-50, 50)}


@pytest.mark.parametrize("name,shift", [(n, s) for n, r in RANGE.items() for s in (r[0], -10, 10, r[1])])
def test_float32_range(tool, name, shift):
    p = _points(name, 3 if name == "gg_ttgg" else 12)
    ref64, ref32 = _run(tool, name, p, "kernels", 173.0)
    v64, v32 = _run(tool, name, np.ldexp(p, shift), "kernels", np.ldexp(173.0, shift))
    back = np.ldexp(1.0, -2 * (4 - p.shape[1]) * shift)
    np.testing.assert_allclose(v64 * back, ref64, rtol=1e-14)
    # exact but for small terms that come out subnormal; 1e-6 is eight units of float32
    np.testing.assert_allclose(v32 * back, ref32, rtol=1e-6)
