"""The table of T(k) of 16-byte plans takes only memory that nothing else needs: requests
fit the budgets that hold their lattices, and the numbers are the same with and without it."""
import pytest

from paper_2006_16935_gb300 import qfd as Q

pytestmark = pytest.mark.gpu


def request(n, prec, kin, seed=3):
    return dict(n=n, a=0.3, mass=1.3, dtau=0.01 if kin != 1 else 0.004, kinetic=kin, nstates=1, precision=prec,
                potential="ho", pot_coeffs=(1.0, 0.0), seed=seed, tol=-1.0, max_steps=120)


def table_bytes(n):
    return 8 * (n // 2 + 1) ** 3


def serve(reqs, budget, **kw):
    with Q.Server(budget, check_every=40, ortho_every=10, **kw) as sv:
        ids = [sv.submit(Q.make_request(**r)) for r in reqs]
        res = sv.run_until_done(len(ids))
    return [res[i] for i in ids]


@pytest.mark.parametrize("n", [16, 64, 96])
@pytest.mark.parametrize("prec", ["c128", "df64", "c64_refine_df"])
@pytest.mark.parametrize("kin", [1, 2, 3])
def test_request_fits_the_budget_of_its_lattices(qfdlib, n, prec, kin):
    tight = serve([request(n, prec, kin)], Q.plan_bytes(n, prec))[0]
    roomy = serve([request(n, prec, kin)], 64e9)[0]
    assert tight["status"] == 0 and roomy["status"] == 0
    assert tight["energy"] == roomy["energy"] and tight["steps"] == roomy["steps"]


@pytest.mark.parametrize("cohorts", [False, True])
def test_tables_make_way_for_a_request(qfdlib, cohorts):
    n, prec = 64, "c128"
    b = Q.plan_bytes(n, prec)
    reqs = [dict(request(n, prec, 2, seed=s), max_steps=2000) for s in (5, 6)]
    with Q.Server(2 * b, check_every=40, ortho_every=10, cohorts=cohorts) as sv:
        ids = [sv.submit(Q.make_request(**reqs[0]))]
        got = {}
        for _ in range(4):  # the first request runs alone, its periods captured, with its table
            got.update((r["id"], r) for r in sv.poll())
        assert sv.stats()["used_bytes"] == b + table_bytes(n)
        ids.append(sv.submit(Q.make_request(**reqs[1])))
        got.update((r["id"], r) for r in sv.poll())
        assert sv.stats()["active"] == 2 and sv.stats()["used_bytes"] == 2 * b
        while len(got) < 2:
            got.update((r["id"], r) for r in sv.poll())
        assert sv.stats()["used_bytes"] == 0
    for req, i in zip(reqs, ids):
        assert got[i]["status"] == 0
        assert got[i]["energy"] == serve([req], 64e9)[0]["energy"]
