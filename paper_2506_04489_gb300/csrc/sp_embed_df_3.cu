// double-float passes of sp_embed.cuh, length group 3, compiled apart to keep translation units small.
#include "sp_embed.cuh"

SP_F_GROUP3(SP_EMBED_DF32, )
