"""A bond that meets entries that are not numbers ends the run (TTC_ERR_NONFINITE) in a
decision in which other bonds take a pivot: their ranks count it, so their pivot
inverses have to have its row and column too.  The entries (a, b, c, :) enter bond
1's superblock with c, the first index behind a pivot of bond 2, and stay out of
the others', a being none of bond 1's pivots.  Checked: U_k P_k = 1 for the
pivots' entries P_k, persistent (in a batch that goes on) and host-stepped.

Tolerance: P_k is a leading block of the pivots' matrix of a TT with terms down
to 0.6^12 = 2e-3 at ranks up to 12: condition below 1e6, so U P is within
1e6 * 12 * 2^-53 = 1.4e-9 of the identity; 1e-6."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

N, NS, CAP, R = [40, 41, 42, 20], 3000, 12, 12


def tensor(a=None):
    r, rng, cores = R + 2, np.random.default_rng(4), []
    for m in range(4):
        c = np.zeros((1 if m == 0 else r, N[m], 1 if m == 3 else r))
        for j in range(R):
            f = np.cos(2 * np.pi * (0.4 * (j + 1) * np.arange(N[m]) / N[m] + rng.random()))
            c[0 if m == 0 else j, :, 0 if m == 3 else j] = f * (0.6 ** j if m == 0 else 1.0)
        if a is not None:  # 1e160 * 1e160 - 1e160 * 1e160, each out of range, at a alone
            for j, v in ((R, 1e160), (R + 1, -1e160)):
                c[0 if m == 0 else j, slice(None) if m == 3 else a[m], 0 if m == 3 else j] = (1e160, 1.0, v, 1.0)[m]
        cores.append(c)
    return {"kind": "tt", "ranks": [1, r, r, r, 1], "cores": cores}


def entry(g, i):
    v = g["cores"][0][0, i[0], :R]
    for m in (1, 2, 3):
        v = v @ g["cores"][m][:R, i[m], :R if m < 3 else 1]
    return v[0]


def inverse_errors(c, g):
    out = []
    for k in (1, 2, 3):
        I, J = c.pivots(k)
        P = np.array([[entry(g, tuple(i) + tuple(j)) for j in J] for i in I])
        U = c.pivot_inverse(k)
        assert U.shape == P.shape
        out.append(float(np.abs(U @ P - np.eye(len(P))).max()))
    return out


@pytest.mark.parametrize("residual", ["recompute", "stored"])
@pytest.mark.parametrize("kind", ["batch", "host_loop", "user"])
def test_inverse_after_a_bond_failed(residual, kind):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2407_11290_gb300 import ttcross as tt

    def cross(g):
        if kind == "user":
            w = [torch.from_numpy(x).cuda() for x in g["cores"]]

            def fn(idx, out):
                i = idx.long()
                v = w[0][0, i[:, 0], :]
                for m in (1, 2, 3):
                    v = (v[:, :, None] * w[m].permute(1, 0, 2)[i[:, m]]).sum(1)
                out.copy_(v[:, 0])
            g = {"kind": "user", "fn": fn}
        return tt.TTCross(N, g, max_rank=CAP, nsamples=NS, seed=3, residual=residual,
                          host_loop=kind == "host_loop")

    clean = cross(tensor())
    clean.run(0.0)
    clean.sync()
    J, I1 = clean.pivots(2)[1][:, 0], set(clean.pivots(1)[0][:, 0])
    z = next(z for z in range(4, 9) if J[z] not in J[:z])
    samples = set(map(tuple, oracle.sample_indices(N, NS, 3)[:, :3]))
    a = next((x, y, int(J[z])) for x in range(1, N[0]) for y in range(N[1])
             if x not in I1 and (x, y, int(J[z])) not in samples)
    g = tensor(a)
    bad = cross(g)
    if kind == "batch":  # beside one that goes on
        tt.run_batch([bad, clean], 0.0)
        clean.sync()
        assert max(inverse_errors(clean, g)) <= 1e-6
    else:
        bad.run(0.0)
    assert bad.sync(allow=(tt.ERR_NONFINITE,)) == tt.ERR_NONFINITE
    r = bad.ranks()
    assert r[1] == z + 1 and r[2] in (z + 1, z + 2), (list(r), z)
    assert max(inverse_errors(bad, g)) <= 1e-6, (list(r), z, inverse_errors(bad, g))
