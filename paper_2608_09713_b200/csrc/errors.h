// The device error word and the statuses its bits become.
#pragma once
#include <stdint.h>

#include "../../include/spsyrk.h"

namespace spsyrk {

// bits of the device error word
enum : uint32_t {
    ERRW_BAD_ROWPTR = 1u,
    ERRW_BAD_COL = 2u,
    ERRW_UNSORTED = 4u,
    ERRW_INTERNAL = 8u,
    ERRW_UPPER = 16u,
    ERRW_BAD_CSR = ERRW_BAD_ROWPTR | ERRW_BAD_COL | ERRW_UNSORTED,
};

// What the caller hears: the input's fault if there is one (`of_columns` where a bad column id is not the matrix's own fault),
// SPSYRK_ERR_INTERNAL if a bounded wait ran out.
inline spsyrk_status_t status_of(uint32_t e, spsyrk_status_t of_columns = SPSYRK_ERR_BAD_CSR) {
    if (e & (ERRW_BAD_ROWPTR | ERRW_UNSORTED | ERRW_UPPER)) return SPSYRK_ERR_BAD_CSR;
    if (e & ERRW_BAD_COL) return of_columns;
    return e ? SPSYRK_ERR_INTERNAL : SPSYRK_OK;
}

}  // namespace spsyrk
