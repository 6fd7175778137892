"""The server's binding keeps its context alive: destroying a server restores
the context's options, so the context must not go first when a program drops
both (at interpreter exit, say)."""
from paper_2002_05200_gb300 import logan


class FakeLib:
    def __init__(self):
        self.calls = []

    def __getattr__(self, name):
        def call(*args):
            if name.endswith("_create"):
                next(a for a in args if hasattr(a, "_obj"))._obj.value = 1
            self.calls.append(name)
            return 0
        return call


def test_the_context_outlives_its_server(monkeypatch):
    fake = FakeLib()
    monkeypatch.setattr(logan, "lib", lambda: fake)
    held = {"ctx": logan.Context(0)}
    held["server"] = logan.Server(held["ctx"], budget_bytes=1 << 20)
    held.pop("ctx")
    held.pop("server")
    order = [c for c in fake.calls if c.endswith("_destroy")]
    assert order == ["logan_server_destroy", "logan_ctx_destroy"]
