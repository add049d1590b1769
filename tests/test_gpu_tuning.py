"""The psi z chunk (planes per psi block) and its autotuner.  The chunk is a tiling
knob: every site's arithmetic is the same whatever its value, so every field
must agree bitwise; the autotuner must leave the state untouched and honour its
cache file."""
import numpy as np
import pytest

import paper_1104_0078_gb300 as F
from paper_1104_0078_gb300 import inputs as I

from gpu_helpers import flb_params, weights_column

pytestmark = pytest.mark.gpu

RAGGED = dict(dim=3, q=19, nx=37, ny=23, nz=19, tau=0.8, kT=1e-4, A=-0.05, B=0.3, K=0.04, M=0.1, integrator=2,
              coupling=3, seed=3)


def _start(s, d, rep=0):
    N = d["nx"] * d["ny"] * d["nz"]
    s.set_fields(rep=rep, psi=I.random_field(N, 0.05, 8 + rep))
    s.set_populations(weights_column(d["q"]) + I.random_deviations(d["q"], N, 2e-3, 7 + rep), rep=rep)


def _fields(s, rep=0):
    psi, u = s.get_psi_u(rep)
    return s.get_populations(rep), psi, u


@pytest.mark.parametrize("q,scheme", [(19, 0), (19, 1), (15, 1)])
def test_zchunk_changes_no_bit(q, scheme):
    d = dict(RAGGED, q=q, scheme=scheme)
    ref = None
    for zc in (64, 1, 3, 8, 19):
        s = F.Solver(flb_params(d))
        _start(s, d)
        s.set_tuning(zc)
        assert s.get_tuning(0) == zc
        s.step(12)
        out = _fields(s)
        if ref is None:
            ref = out
        else:
            for a, b in zip(ref, out):
                assert np.array_equal(a, b), zc


def test_batched_with_mixed_zchunks_equals_plain():
    shapes = [(16, 16, 16), (12, 10, 20), (40, 18, 9), (33, 7, 70)]
    ds = [dict(RAGGED, nx=nx, ny=ny, nz=nz, scheme=1, kT=1e-5 * (1 + r), seed=100 + r)
          for r, (nx, ny, nz) in enumerate(shapes)]
    ps = [flb_params(d) for d in ds]
    runs = []
    for mode, chunks in ((F.FLB_MODE_PLAIN, (64, 64, 64, 64)), (F.FLB_MODE_BATCHED, (4, 7, 64, 16))):
        s = F.Solver(ps)
        for r, d in enumerate(ds):
            _start(s, d, r)
            s.set_tuning(chunks[r], rep=r)
        s.set_mode(mode)
        s.step(6)
        s.set_tuning(5, rep=3)              # a change between calls rebuilds the batched graph
        s.step(3)
        runs.append([_fields(s, r) for r in range(len(ps))])
    for ra, rb in zip(*runs):
        for a, b in zip(ra, rb):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("mode", [0, 1])
def test_autotune_keeps_state_and_uses_cache(tmp_path, mode):
    cache = str(tmp_path / "tune.txt")
    d = dict(RAGGED, scheme=1)
    ps = [flb_params(d), flb_params(dict(d, nx=20, ny=20, nz=40, seed=9))]
    s = F.Solver(ps)
    for r in range(2):
        _start(s, dict(d, nx=ps[r].nx, ny=ps[r].ny, nz=ps[r].nz), r)
    s.set_mode(mode)
    s.step(2)
    before = [_fields(s, r) for r in range(2)] + [s.get_step(0)]
    chosen = s.autotune(cache=cache)
    after = [_fields(s, r) for r in range(2)] + [s.get_step(0)]
    for a, b in zip(before[:2], after[:2]):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
    assert before[2] == after[2] == 2
    lines = open(cache).read().splitlines()
    if mode == F.FLB_MODE_BATCHED:
        # one shared value, then one per box depth: a listed value or an even split ceil(nz / k)
        for c, p in zip(chosen, ps):
            assert c in (4, 8, 16, 32, 64) or any(c == -(-p.nz // k) for k in range(1, 17))
        assert len(lines) == 1 + len({p.nz for p in ps})
    else:
        assert all(c in (4, 8, 16, 32, 64) for c in chosen)
        assert len(lines) == 2
    # a second handle of the same configuration takes the cached values without timing
    s2 = F.Solver(ps)
    s2.set_mode(mode)
    assert s2.autotune(cache=cache) == chosen
    assert open(cache).read().splitlines() == lines
    # forcing re-times and appends; the state still steps on identically
    s2.autotune(cache=cache, force=True)
    assert len(open(cache).read().splitlines()) == 2 * len(lines)
    s.step(3)
    ref = F.Solver(ps)
    for r in range(2):
        _start(ref, dict(d, nx=ps[r].nx, ny=ps[r].ny, nz=ps[r].nz), r)
    ref.step(5)
    for r in range(2):
        for x, y in zip(_fields(s, r), _fields(ref, r)):
            assert np.array_equal(x, y)


def test_tuning_argument_checks():
    s = F.Solver(flb_params(dict(RAGGED, scheme=1)))
    for bad in (0, -3, 5000):
        with pytest.raises(F.FlbError):
            s.set_tuning(bad)
    with pytest.raises(F.FlbError):
        s.set_tuning(8, rep=3)


@pytest.mark.parametrize("q,scheme", [(19, 0), (15, 0), (19, 1)])
def test_autotune_of_the_single_pass_step(tmp_path, q, scheme):
    # the single-pass step has a depth under the FD scheme too, whose two-launch form has none
    cache = str(tmp_path / "tune.txt")
    p = flb_params(dict(RAGGED, q=q, scheme=scheme))
    s = F.Solver(p)
    assert s.get_tuning(0) == 64
    s.set_psi_fused(True)
    (chosen,) = s.autotune(cache=cache)
    assert chosen in (4, 8, 16, 32)  # the candidates up to the first that covers 19 planes
    lines = open(cache).read().splitlines()
    assert len(lines) == 1 and lines[0].endswith(f"\t{chosen}")
    s.set_psi_fused(False)
    assert s.get_tuning(0) == 64     # the two-launch form keeps its own
    s2 = F.Solver(p)
    s2.set_psi_fused(True)
    assert s2.autotune(cache=cache) == [chosen]
    assert open(cache).read().splitlines() == lines


def _planes(s, fused=False):
    s.set_psi_fused(fused)
    return s.get_psi_planes(0)


def test_cache_keeps_the_tuned_form(tmp_path):
    # a cached handle runs the form that its line names, small tiles or planes, whatever its size
    cache = tmp_path / "tune.txt"
    p = flb_params(dict(RAGGED, scheme=1))
    s = F.Solver(p)
    assert s.get_psi_planes(0) == 0                          # by its size
    (chosen,) = s.autotune(cache=str(cache))
    key, planes, form = cache.read_text().rstrip("\n").split("\t")
    assert int(planes) == chosen and form in "01"
    assert s.get_psi_planes(0) == (0 if form == "1" else chosen)
    for form, runs in (("0", 8), ("1", 0)):
        cache.write_text(f"{key}\t8\t{form}\n")
        s = F.Solver(p)
        assert s.autotune(cache=str(cache)) == [8]
        assert s.get_psi_planes(0) == runs
    assert cache.read_text().count("\n") == 1               # both without timing
    # the single-pass step is another configuration, and its tuning leaves the tiles as they are
    s.set_psi_fused(True)
    (one,) = s.autotune(cache=str(cache))
    assert cache.read_text().count("\n") == 2
    assert _planes(s, True) == one and _planes(s) == 0


@pytest.mark.parametrize("other", [dict(storage=F.FLB_F16_DEV), dict(force_grad=F.FLB_FORCE_STRESS), dict(coupling=2)])
@pytest.mark.parametrize("mode", [0, 1])
def test_cache_separates_configurations_of_other_kernels(tmp_path, mode, other):
    # FP16 storage draws by other normals, and without a given mu stage 1 is another kernel
    cache = tmp_path / "tune.txt"
    lines = []
    for d in (dict(RAGGED, scheme=1), dict(RAGGED, scheme=1, **other)):
        s = F.Solver(flb_params(d))
        s.set_mode(mode)
        s.autotune(cache=str(cache))
        lines.append(cache.read_text().count("\n"))
    assert lines[1] == 2 * lines[0]


def test_planes_in_use():
    s = F.Solver(flb_params(dict(RAGGED, scheme=1)))
    assert s.get_psi_planes(0) == 0
    s.set_tuning(7)
    assert s.get_psi_planes(0) == 7
    s.set_mode(F.FLB_MODE_BATCHED)
    assert s.get_psi_planes(0) == 7
    s = F.Solver(flb_params(dict(RAGGED, scheme=0)))
    s.set_tuning(7)                                          # FD: the single-pass step's alone
    assert _planes(s) == 0 and _planes(s, True) == 7
    with pytest.raises(F.FlbError):
        s.get_psi_planes(1)


def test_modes_keep_their_own_depth(tmp_path):
    cache = tmp_path / "tune.txt"
    p = flb_params(dict(RAGGED, scheme=1))

    def tuned(mode):
        s.set_mode(mode)
        return s.autotune(cache=str(cache))

    s = F.Solver(p)
    tuned(F.FLB_MODE_PLAIN)
    tuned(F.FLB_MODE_BATCHED)
    lines = [l.split("\t")[0] for l in cache.read_text().splitlines()]
    plain = [k for k in lines if k.startswith("plain|")]
    assert len(plain) == 1 and len(lines) > 1
    cache.write_text("".join(k + ("\t8\t0\n" if k in plain else "\t5\n") for k in lines))
    s = F.Solver(p)
    assert tuned(F.FLB_MODE_PLAIN) == [8]
    assert tuned(F.FLB_MODE_BATCHED) == [5]
    assert (s.get_tuning(0), s.get_psi_planes(0)) == (5, 5)
    s.set_mode(F.FLB_MODE_PLAIN)
    assert (s.get_tuning(0), s.get_psi_planes(0)) == (8, 8)
    s.set_mode(F.FLB_MODE_PERSISTENT)
    assert (s.get_tuning(0), s.get_psi_planes(0)) == (5, 5)


@pytest.mark.parametrize("integrator", [1, 2])
def test_autotune_times_both_groups_of_a_large_ensemble(integrator):
    # from 600 thousand sites on a step launches the stages of two groups of replicas; at a depth
    # of 4 the chunks 4, 2 and 1 are timed, each in four runs
    ps = [flb_params(dict(RAGGED, nx=320, ny=317, nz=4, scheme=1, integrator=integrator, seed=r)) for r in range(2)]
    s = F.Solver(ps)
    s.set_mode(F.FLB_MODE_BATCHED)
    before = s.launch_count()
    chosen = s.autotune()
    assert set(chosen) <= {1, 2, 4}
    assert s.launch_count() - before == 3 * 4 * integrator * 2
