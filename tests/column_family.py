"""Which family the default adjoint takes for a call, without a GPU fault or
an entry point of its own: only the column form asks for a workspace once the
geometry's tables exist, so it uses up an allocation failure that was set."""
import torch


def takes_columns(gjp, proj, g, vg) -> bool:
    """Whether ``gjp.adjoint(proj, g, vg.n, vg.h, vg.origin)`` takes the column form."""
    from paper_1609_00958_gb300 import _capi
    gjp.adjoint(proj, g, vg.n, vg.h, vg.origin)              # tables and column records
    fresh = gjp.Geometry([[9.0, 0.0, 0.0]], [[-9.0, 0.0, 0.0]], [[0.0, 1.0, 0.0]], [[0.0, 0.0, 1.0]], 1, 1)
    vol = torch.zeros((2, 2, 2), device="cuda")
    try:
        assert _capi.gjp_debug_fail_allocations(1) == _capi.GJP_OK
        gjp.adjoint(proj, g, vg.n, vg.h, vg.origin)
        try:
            gjp.forward(vol, fresh, (1.0, 1.0, 1.0))         # its table takes the failure if the adjoint did not
        except gjp.GjpError:
            return False
        return True
    finally:
        _capi.gjp_debug_fail_allocations(0)
