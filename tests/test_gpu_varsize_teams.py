"""The warp teams of an uneven batch's persistent launch: the methods and systems
that still take them, at every team size, staging and block shape."""

import numpy as np
import pytest

import oracle
from paper_2308_08417_gb300 import workloads as W
from tests.parity import compare
from tests.test_gpu_varsize import run_plan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bbs():
    from paper_2308_08417_gb300 import _build, bbs as mod

    _build.build()
    return mod


@pytest.fixture(scope="module")
def handle(bbs):
    return bbs.Handle(0)


def perturbed(vb, seed):
    rng = np.random.default_rng(seed)
    return W.VarBatch(vb.patterns, vb.sys_pattern, vb.val_off, vb.vec_off,
                      vb.values * (1.0 + 1e-15 * rng.uniform(-1.0, 1.0, vb.values.shape)), vb.b, vb.x0, vb.name)


def check(vb, got, idx, **kw):
    """The parity bar; counts within 2 plus the oracle's own range when the values
    are perturbed at rounding level."""
    xr, itr, _, sr = oracle.solve_varsize(vb, systems=idx, **kw)
    its = np.array([np.asarray(oracle.solve_varsize(perturbed(vb, s), systems=idx, **kw)[1], dtype=np.int64)
                    for s in range(1, 9)])
    tol = 2 + its.max(axis=0) - its.min(axis=0)
    fails = []
    for k, i in enumerate(idx):
        o, n = int(vb.vec_off[i]), int(vb.sys_n()[i])
        fails += compare(got[0][None, o:o + n], got[1][i:i + 1], got[2][i:i + 1], got[3][i:i + 1], xr[None, o:o + n],
                         itr[k:k + 1], sr[k:k + 1], iter_tol=tol[k], label=f"system {i} (n={n}) {kw}")
    assert not fails, "\n".join(fails[:10])


def explicit(bbs, bw, stage, max_n=1024):
    t = bbs.bbs_var_default_tuning(max_n)
    t.block_warps = bw
    for k in range(t.num_buckets):
        t.stage_values[k] = stage
        t.team_warps[k] = min(bw, 2 ** k // 2 or 1)
        t.pack[k] = t.wide[k] = 0
    return t


@pytest.mark.parametrize("kw", [dict(solver="cg"), dict(precond="none")])
def test_team_sizes_staging_and_block_shapes(bbs, handle, kw):
    vb = W.uneven(700, n_max=900)
    if kw.get("solver") == "cg":
        for pi, p in enumerate(vb.patterns):
            members = np.nonzero(vb.sys_pattern == pi)[0]
            if len(members):
                vals = W.stencil_values(p, len(members), np.random.default_rng(pi), 0.05, 0.5, symmetric=True)
                for k, i in enumerate(members):
                    vb.values[int(vb.val_off[i]):int(vb.val_off[i]) + p.nnz] = vals[k]
    vbd = bbs.VarDeviceBatch.from_varbatch(vb)
    idx = np.random.default_rng(3).choice(vb.num_batch, 90, replace=False)
    for bw in (8, 16):
        for stage in (0, 1):
            plan = bbs.VarPlan(handle, vbd, bbs.bbs_default_options(**kw), explicit(bbs, bw, stage))
            d = plan.describe()
            assert d["team_systems"] == vb.num_batch and d["persistent_grid"] > 0
            check(vb, run_plan(bbs, plan, vb), idx, **kw)


@pytest.mark.parametrize("bw", [8, 16])
def test_systems_too_dense_to_stage_beside_ordinary_ones(bbs, handle, bw):
    """BiCGSTAB with Jacobi: full systems of n = 190 (289 KB of values) stay with the
    warp teams, in the same plan as stencils in packed, block and wide launches."""
    vb = W.uneven(300, n_max=900)
    rng = np.random.default_rng(5)
    full = W.random_pattern(190, 190 * 190, rng)
    count = 12
    vals = W.general_values(full, count, rng, 0.05, 0.5)
    b = rng.uniform(-1, 1, (count, full.n))
    vec_off = np.concatenate([vb.vec_off, len(vb.b) + full.n * np.arange(count)])
    val_off = np.concatenate([vb.val_off, len(vb.values) + full.nnz * np.arange(count)])
    index = np.concatenate([vb.sys_pattern, np.full(count, len(vb.patterns), dtype=np.int32)]).astype(np.int32)
    both = W.VarBatch(list(vb.patterns) + [full], index, val_off, vec_off, np.concatenate([vb.values, vals.ravel()]),
                      np.concatenate([vb.b, b.ravel()]), np.zeros(len(vb.b) + b.size), "mixed")
    vbd = bbs.VarDeviceBatch.from_varbatch(both)
    t = bbs.bbs_var_default_tuning(1024)
    t.block_warps = bw
    plan = bbs.VarPlan(handle, vbd, bbs.bbs_default_options(), t)
    d = plan.describe()
    assert d["team_systems"] > count and d["packed_systems"] > 0
    got = run_plan(bbs, plan, both)
    assert (got[3] == 0).all()
    check(both, got, np.concatenate([np.arange(0, 300, 4), 300 + np.arange(count)]))


def test_tuner_leaves_choices_without_effect(bbs, handle):
    """BiCGSTAB with Jacobi and systems that blocks can stage: team warps, staging
    and block warps reach no launch, and come back as the default's."""
    import torch

    vb = W.uneven(1500)
    vbd = bbs.VarDeviceBatch.from_varbatch(vb)
    tuned = bbs.bbs_var_tune(handle, vbd, torch.as_tensor(vb.b, device="cuda"), torch.as_tensor(vb.x0, device="cuda"),
                             bbs.bbs_default_options(), sample=96).as_dict()
    want = bbs.bbs_var_default_tuning(int(vb.sys_n().max())).as_dict()
    for key in ("team_warps", "stage_values", "block_warps"):
        assert tuned[key] == want[key], key


@pytest.mark.parametrize("kw", [dict(), dict(solver="cg"), dict(precond="none")])
def test_packed_sizes_at_the_edges_of_their_classes(bbs, handle, kw):
    """n = 3 and every multiple of 16 with its neighbours up to 160, with Jacobi in
    ten classes of 16 lanes (few codes at once; narrower groups, 4 and 8 lanes too,
    without a preconditioner)."""
    rng = np.random.default_rng(17)
    sizes = [3] + sorted({n for k in range(1, 11) for n in (16 * k - 1, 16 * k, 16 * k + 1) if n <= 160})
    pats = [W.stencil_pattern("1d3", n) for n in sizes]
    index = np.tile(np.arange(len(pats), dtype=np.int32), 11)
    vals = [W.stencil_values(pats[p], 1, rng, 0.05, 0.5, symmetric=True)[0] for p in index]
    n = np.array([pats[p].n for p in index])
    nnz = np.array([pats[p].nnz for p in index])
    b = rng.uniform(-1, 1, int(n.sum()))
    vb = W.VarBatch(pats, index, np.cumsum(nnz) - nnz, np.cumsum(n) - n, np.concatenate(vals), b, np.zeros(len(b)),
                    "edges")
    plan = bbs.VarPlan(handle, bbs.VarDeviceBatch.from_varbatch(vb), bbs.bbs_default_options(**kw))
    d = plan.describe()
    assert d["packed_systems"] == vb.num_batch
    assert d["packed_launches"] == 10 or "precond" in kw and d["packed_launches"] > 10
    got = run_plan(bbs, plan, vb)
    assert (got[3] == 0).all()
    check(vb, got, np.arange(0, vb.num_batch, 2), **kw)
