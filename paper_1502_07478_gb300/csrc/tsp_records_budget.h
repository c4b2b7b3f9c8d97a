// Device memory that the window records may take.
#pragma once

#include <cstddef>

// A quarter of what would be free without records, the records of a batch's other
// members among them (`others`, in bytes, held): 6e7 events at 1 mm on an empty 280 GB.
// avail: free now, the context's own old buffer counted as free.
inline bool records_allowed(size_t need, size_t others, size_t avail)
{
    return need + others <= (avail + others) / 4;
}
