"""The cost model rates a specialised candidate by the program that its apply
runs, which its statistics have then compiled (host only)."""
import synth


def test_specialised_candidates_are_rated_by_their_own_program(monkeypatch):
    from paper_2205_06973_gb300 import build
    build.build()
    from paper_2205_06973_gb300 import api, autotune
    asked = []
    stats = api.Plan.stats

    def spy(self, *a, **k):
        asked.append((self.method, self.k, bool(k.get("jit"))))
        return stats(self, *a, **k)

    monkeypatch.setattr(api.Plan, "stats", spy)
    n = 29
    plan, tc, est, jit = autotune.choose_plan(synth.qft(n), n)
    assert [(m, k, j) for m, k, j in asked] == [(c[0], c[1], c[3]) for c in autotune.PLAN_CANDIDATES]
    assert jit == [e for e in est if e["est_s"] == min(x["est_s"] for x in est)][0]["jit"]
    plan.close()
